// cells.cu -- staging of FP64 state into the dense kernels' mirrors, the hashed
// cell list, and force assembly (Sec. 3.1, step 2: F_ext + pair interactions,
// the primed sums accelerated by neighbour lists; the paper notes that particle
// sorting is needed for these short-ranged parts but not for the all-pairs sum,
// Sec. 3.2).
//
// Cell list: cells of side h >= max(r_near, repulsion cutoff) over FP64
// positions; the integer cell (cx, cy, cz) is hashed into H = 2^k >= 2n buckets,
// so unbounded domains need no bounding box.  Build = count, exclusive scan,
// scatter, and an insertion sort of each bucket by particle index (makes every
// neighbour walk, hence every FP64 near-pair sum, independent of atomics order).
#include <algorithm>
#include <type_traits>

#include "neighbours.cuh"

namespace sd {

// ---------------------------------------------------------------- staging

template <typename V4>
__global__ void stage_pos_kernel(const double *__restrict__ x, V4 *__restrict__ m, float *__restrict__ soa, int n,
                                 int npad, Box b, int *err) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double px = x[3 * i], py = x[3 * i + 1], pz = x[3 * i + 2];
    if (!isfinite(px) || !isfinite(py) || !isfinite(pz)) atomicOr(err, DEV_ERR_NONFINITE);
    put_pos_mirror(m, soa, npad, i, x, b);
}

cudaError_t launch_stage_pos(sd_handle *h, cudaStream_t st, const double *x64, Mirror posm) {
    if (h->n == 0) return cudaSuccess;
    const int nb = (h->n + 255) / 256;
    if (h->mode == MODE_FP64)
        stage_pos_kernel<dbl4><<<nb, 256, 0, st>>>(x64, static_cast<dbl4 *>(posm.aos), posm.soa, h->n, h->npad,
                                                   h->cl.box, h->d_err);
    else
        stage_pos_kernel<float4><<<nb, 256, 0, st>>>(x64, static_cast<float4 *>(posm.aos), posm.soa, h->n, h->npad,
                                                     h->cl.box, h->d_err);
    ++h->launches;
    return cudaGetLastError();
}

// The Verlet step's first kernel: the mirror of x (as the cell-list build writes it),
// the rebuild decision and the clamp flag of the step, both written by the last block
// to finish (vl[0] and *flag; vl[1] counts the blocks, vl[2] gathers their bits).
//   * The list holds the pairs within r_near + skin of the positions xref it was
//     built from.  While every particle's displacement since then, relative to
//     particle 0's, stays below skin / 2, pair distances have changed by less than
//     the skin (a uniform translation moves no pair), so the list still holds every
//     pair within r_near.  It is rebuilt early, from skin / 4 on, so that this holds
//     in the step that rebuilds it too.
//   * The clamp flag (some pair closer than r_safe: the all-pairs kernel then clamps
//     every tile) comes from the pairs of that list, in FP64 exactly as the near pass
//     tests them, so the all-pairs kernel need not wait for the near pass.  It is
//     raised outright when the list may miss pairs: no list yet (bit 2 of vl[0]:
//     positions never set), overflowed (its particles corrected in place), or a
//     displacement of skin / 2 or more.  (The list is the steps' own, built by the
//     first step after the positions are set and by the steps' rebuilds; no other pass touches it.)
// A thread takes particles and listed pairs in turn over a grid that reaches every SM: one
// thread walking a particle's run, in CTAs of 256, took 12 us (N = 4,096) to 17 us (4,913
// on a lattice); now 8 and 9 us, cold caches.
template <typename V4>
__global__ void __launch_bounds__(128) verlet_check_kernel(const double *__restrict__ x, const double *__restrict__ xref,
                                                           int n, int npad, Box b, double quarter_skin2,
                                                           double half_skin2, double rsafe2, V4 *__restrict__ m,
                                                           float *__restrict__ soa, int *flag, int *vl,
                                                           const unsigned long long *near_n, int cap,
                                                           const int2 *__restrict__ ent, int *err) {
    const long long gt = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x,
                    stride = static_cast<long long>(gridDim.x) * blockDim.x;
    const unsigned long long listed = *near_n;
    // 1: rebuild; 2: clamp every tile (vl[0] is written below, after every block has read it)
    int bits = (*static_cast<volatile int *>(vl) & 2) || listed > static_cast<unsigned long long>(cap) ? 3 : 0;
    const long long work = n + (bits ? 0 : static_cast<long long>(listed));   // (a raised clamp bit needs no pairs)
    for (long long q = gt; q < work; q += stride) {
        if (q < n) {
            const long long i = q;
            const double px = x[3 * i], py = x[3 * i + 1], pz = x[3 * i + 2];
            if (!isfinite(px) || !isfinite(py) || !isfinite(pz)) atomicOr(err, DEV_ERR_NONFINITE);
            put_pos_mirror(m, soa, npad, static_cast<int>(i), x, b);
            const double ux = (px - xref[3 * i]) - (x[0] - xref[0]);
            const double uy = (py - xref[3 * i + 1]) - (x[1] - xref[1]);
            const double uz = (pz - xref[3 * i + 2]) - (x[2] - xref[2]);
            const double u2 = ux * ux + uy * uy + uz * uz;
            if (!(u2 < quarter_skin2)) bits |= 1;   // (also NaN)
            if (!(u2 < half_skin2)) bits |= 3;
        } else {
            const int2 p = ent[q - n];
            const int i = static_cast<int>(dbg_index(p.x, n, err)), j = static_cast<int>(dbg_index(p.y, n, err));
            if (i > j) continue;   // (both orders are listed)
            double dx = x[3 * i] - x[3 * j], dy = x[3 * i + 1] - x[3 * j + 1], dz = x[3 * i + 2] - x[3 * j + 2];
            box_image(b, dx, dy, dz);
            if (dx * dx + dy * dy + dz * dz < rsafe2) bits |= 2;
        }
    }
    const int any = (__syncthreads_or(bits & 1) ? 1 : 0) | (__syncthreads_or(bits & 2) ? 2 : 0);
    if (threadIdx.x == 0) {
        if (any) atomicOr(&vl[2], any);
        __threadfence();
        const int done = atomicAdd(&vl[1], 1);
        if (done == static_cast<int>(gridDim.x) - 1) {   // every block's bits are in
            __threadfence();
            const int all = atomicExch(&vl[2], 0);
            *flag = (all & 2) ? 1 : 0;
            vl[0] = all & 1;
            vl[1] = 0;
        }
    }
}

cudaError_t launch_verlet_check(sd_handle *h, cudaStream_t st, const double *x64, Mirror posm) {
    if (h->n == 0) return cudaSuccess;
    const int nb = static_cast<int>(std::min<long long>((static_cast<long long>(h->n) * 4 + 127) / 128, 4LL * h->num_sms));
    const double hs2 = 0.25 * h->skin * h->skin, qs2 = 0.0625 * h->skin * h->skin;
    const double rs2 = kRSafe * kRSafe * h->pc.a * h->pc.a;
    prof_begin(h, SD_KERNEL_CELLS, st);
    if (h->mode == MODE_FP64)
        verlet_check_kernel<dbl4><<<nb, 128, 0, st>>>(x64, h->xref, h->n, h->npad, h->cl.box, qs2, hs2, rs2,
                                                      static_cast<dbl4 *>(posm.aos), posm.soa, h->d_flag, h->d_vl,
                                                      h->vn, h->near_cap, h->vent, h->d_err);
    else
        verlet_check_kernel<float4><<<nb, 128, 0, st>>>(x64, h->xref, h->n, h->npad, h->cl.box, qs2, hs2, rs2,
                                                        static_cast<float4 *>(posm.aos), posm.soa, h->d_flag, h->d_vl,
                                                        h->vn, h->near_cap, h->vent, h->d_err);
    prof_end(h, SD_KERNEL_CELLS, st);
    ++h->launches;
    return cudaGetLastError();
}

// dst64 = src (+ fext + gravity when add_ext) and its mirror; src is n x 3 float or double.
// A second array (src2, without fext) rides along as the grid's second row.
template <typename V4, typename Src>
__global__ void stage_forces_kernel(const Src *__restrict__ src, const double *__restrict__ fext, double gx,
                                    double gy, double gz, double *__restrict__ dst, V4 *__restrict__ m,
                                    float *__restrict__ soa, const Src *__restrict__ src2, double *__restrict__ dst2,
                                    V4 *__restrict__ m2, float *__restrict__ soa2, int n, int npad, int *err) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (blockIdx.y) {
        src = src2;
        fext = nullptr;
        dst = dst2;
        m = m2;
        soa = soa2;
    }
    double f[3];
    for (int d = 0; d < 3; ++d) f[d] = src ? static_cast<double>(src[3 * i + d]) : 0.0;
    if (fext) {
        f[0] += fext[3 * i] + gx;
        f[1] += fext[3 * i + 1] + gy;
        f[2] += fext[3 * i + 2] + gz;
    }
    if (!isfinite(f[0]) || !isfinite(f[1]) || !isfinite(f[2])) atomicOr(err, DEV_ERR_NONFINITE);
    dst[3 * i] = f[0];
    dst[3 * i + 1] = f[1];
    dst[3 * i + 2] = f[2];
    put_mirror(m, soa, npad, i, f[0], f[1], f[2]);
}

template <typename V4, typename Src>
static void stage_forces_launch(sd_handle *h, cudaStream_t st, const void *src, const double *fe, double *dst64,
                                Mirror dstm, const void *src2, double *dst2, Mirror dstm2) {
    const dim3 nb((h->n + 255) / 256, src2 ? 2 : 1);
    const double *g = h->cfg.gravity;
    stage_forces_kernel<V4, Src><<<nb, 256, 0, st>>>(static_cast<const Src *>(src), fe, g[0], g[1], g[2], dst64,
                                                     static_cast<V4 *>(dstm.aos), dstm.soa,
                                                     static_cast<const Src *>(src2), dst2, static_cast<V4 *>(dstm2.aos),
                                                     dstm2.soa, h->n, h->npad, h->d_err);
}

// src_dtype: SD_DTYPE_F32 / SD_DTYPE_F64 (src may be NULL = zeros); add_ext: add
// the handle's F_ext and gravity.
cudaError_t launch_stage_forces(sd_handle *h, cudaStream_t st, const void *src, int src_dtype, int add_ext,
                                double *dst64, Mirror dstm, const void *src2, double *dst2, Mirror dstm2) {
    if (h->n == 0) return cudaSuccess;
    const double *fe = add_ext ? h->fext64 : nullptr;
    if (h->mode == MODE_FP64) {
        if (src_dtype == SD_DTYPE_F32) stage_forces_launch<dbl4, float>(h, st, src, fe, dst64, dstm, src2, dst2, dstm2);
        else stage_forces_launch<dbl4, double>(h, st, src, fe, dst64, dstm, src2, dst2, dstm2);
    } else {
        if (src_dtype == SD_DTYPE_F32) stage_forces_launch<float4, float>(h, st, src, fe, dst64, dstm, src2, dst2, dstm2);
        else stage_forces_launch<float4, double>(h, st, src, fe, dst64, dstm, src2, dst2, dstm2);
    }
    ++h->launches;
    return cudaGetLastError();
}

// Padding entries n..npad-1 of a position mirror: far from every particle
// (1e18, 0, 0), so that with their zero padding force each pair term with them is
// exactly zero even where the all-pairs kernel does not clamp r^2.
template <typename V4>
__global__ void pad_mirror_kernel(V4 *__restrict__ m, float *__restrict__ soa, int n, int npad) {
    const int i = n + blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npad) return;
    put_mirror(m, soa, npad, i, 1.0e18, 0.0, 0.0);
}

cudaError_t launch_pad_mirror(sd_handle *h, cudaStream_t st, Mirror m) {
    const int npad = h->npad > 0 ? h->npad : kPadTo;
    const int cnt = npad - h->n;
    if (cnt <= 0) return cudaSuccess;
    const int nb = (cnt + 255) / 256;
    if (h->mode == MODE_FP64)
        pad_mirror_kernel<dbl4><<<nb, 256, 0, st>>>(static_cast<dbl4 *>(m.aos), m.soa, h->n, npad);
    else
        pad_mirror_kernel<float4><<<nb, 256, 0, st>>>(static_cast<float4 *>(m.aos), m.soa, h->n, npad);
    ++h->launches;
    return cudaGetLastError();
}

// ---------------------------------------------------------------- cell list

// Bins particle i and writes its mirror (position relative to particle 0, in the
// dense kernels' precision), so the mirror is a pure function of the FP64 state.  A
// Verlet list's build (xref given) records the positions in xref too and leaves the
// clamp flag to the step's check kernel; it needs the mirror of these positions, since the
// list's candidates are screened on it and no step may have written it since they moved.
template <typename V4>
__global__ void cells_hash_kernel(const double *__restrict__ x, int n, CellList c, V4 *__restrict__ m,
                                  float *__restrict__ soa, int npad, int *flag, unsigned long long *near_n,
                                  double *__restrict__ xref, int *vl, int *err) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (i == 0) {
        *near_n = 0;            // the near pass fills its candidate list from the start
        if (xref) vl[0] = 0;    // (there is a list)
        else *flag = 0;         // ... and raises the flag again if needed
    }
    const double px = x[3 * i], py = x[3 * i + 1], pz = x[3 * i + 2];
    if (xref) {
        xref[3 * i] = px;
        xref[3 * i + 1] = py;
        xref[3 * i + 2] = pz;
    }
    if (!isfinite(px) || !isfinite(py) || !isfinite(pz)) atomicOr(err, DEV_ERR_NONFINITE);
    put_pos_mirror(m, soa, npad, i, x, c.box);
    bin_particle(c, i, px, py, pz);
}

constexpr int kScanThreads = 1024;
constexpr int kScanBlock = kScanThreads * kScanPer;   // buckets one scan block covers (one kernel up to this)

__global__ void __launch_bounds__(kScanThreads) scan_blocks_kernel(const int *__restrict__ in, int *__restrict__ out,
                                                                   int *__restrict__ bsum, int H) {
    __shared__ int s_warp[33];
    const int base = blockIdx.x * kScanBlock + threadIdx.x * kScanPer;
    int v[kScanPer];
    scan_load(in, base, H, v);
    const int total = block_exclusive_scan<kScanThreads>(v, s_warp);
    scan_store(out, base, H, v);
    if (threadIdx.x == 0) {
        bsum[blockIdx.x] = total;
        if (gridDim.x == 1) out[H] = total;   // one block: the scan is complete
    }
}

// One block: exclusive scan of the block totals in place (nblk <= kScanBlock
// per pass, looping with a carry), then start[H] = grand total.
__global__ void __launch_bounds__(kScanThreads) scan_top_kernel(int *__restrict__ bsum, int nblk,
                                                                int *__restrict__ start, int H) {
    __shared__ int s_warp[33];
    int carry = 0;
    for (int b0 = 0; b0 < nblk; b0 += kScanBlock) {
        const int base = b0 + threadIdx.x * kScanPer;
        int v[kScanPer];
        for (int k = 0; k < kScanPer; ++k) v[k] = (base + k < nblk) ? bsum[base + k] : 0;
        const int total = block_exclusive_scan<kScanThreads>(v, s_warp);
        for (int k = 0; k < kScanPer; ++k)
            if (base + k < nblk) bsum[base + k] = v[k] + carry;
        carry += total;
    }
    if (threadIdx.x == 0) start[H] = carry;
}

__global__ void scan_add_kernel(int *__restrict__ start, const int *__restrict__ bsum, int H) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < H) start[e] += bsum[e / kScanBlock];
}

__global__ void cells_scatter_kernel(const uint32_t *__restrict__ key, int n, const int *__restrict__ start,
                                     int *__restrict__ cnt, int *__restrict__ sorted, int *err) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) scatter_particle(key, start, cnt, sorted, i, err);
}

__global__ void cells_sort_kernel(const int *__restrict__ start, int *__restrict__ sorted, int H) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < H) sort_bucket(start, sorted, b);
}

cudaError_t launch_build_cells(sd_handle *h, cudaStream_t st, const double *x64, Mirror posm, double *xref) {
    CellList &c = h->cl;
    if (h->n == 0) return cudaSuccess;
    prof_begin(h, SD_KERNEL_CELLS, st);
    // (the bucket counters are zero: zeroed at creation, counted back to zero by
    // every build's scatter)
    const int nb = (h->n + 255) / 256;
    if (h->mode == MODE_FP64)
        cells_hash_kernel<dbl4><<<nb, 256, 0, st>>>(x64, h->n, c, static_cast<dbl4 *>(posm.aos), posm.soa, h->npad,
                                                    h->d_flag, xref ? h->vn : h->near_n, xref, h->d_vl, h->d_err);
    else
        cells_hash_kernel<float4><<<nb, 256, 0, st>>>(x64, h->n, c, static_cast<float4 *>(posm.aos), posm.soa, h->npad,
                                                      h->d_flag, xref ? h->vn : h->near_n, xref, h->d_vl, h->d_err);
    const int nblk = (c.H + kScanBlock - 1) / kScanBlock;
    scan_blocks_kernel<<<nblk, kScanThreads, 0, st>>>(c.cnt, c.start, c.bsum, c.H);
    if (nblk > 1) {
        scan_top_kernel<<<1, kScanThreads, 0, st>>>(c.bsum, nblk, c.start, c.H);
        scan_add_kernel<<<(c.H + 255) / 256, 256, 0, st>>>(c.start, c.bsum, c.H);
        h->launches += 2;
    }
    cells_scatter_kernel<<<nb, 256, 0, st>>>(c.key, h->n, c.start, c.cnt, c.sorted, h->d_err);
    cells_sort_kernel<<<(c.H + 255) / 256, 256, 0, st>>>(c.start, c.sorted, c.H);
    prof_end(h, SD_KERNEL_CELLS, st);
    h->launches += 4;
    return cudaGetLastError();
}

// A Verlet step's rebuild, if its check asked for one, in one launch: bin, scan, scatter and
// sort by one cluster, its CTAs meeting at the hardware barrier.  Rebuilds are rare, and
// what counts is the launch that returns at once: as four to six kernels they cost every
// step 2 to 3 us each.  CTAs of 256, because the launch
// shares the GPU with the all-pairs kernel: 1,024 threads found room only after it.  (A
// cooperative kernel over all SMs costs some 20 us as a graph node; a build that is certain
// to run takes the kernels above, faster from N = 16,384 on and as fast below.)
// What bounds it is a chain of L2 latencies, so a thread's particles and buckets are taken four at
// a time, their loads and atomics in flight together, and scans move 16 bytes an access: N = 4,096
// / 16,384 / 32,768 24 / 47 / 84 us one at a time, now 16 / 30 / 51 (cold caches).  The separate
// kernels take 17 / 25 / 26, of which a step that needs none would pay three to five more launches.
// Eight at a time are no faster and take 80 registers instead of 64.
constexpr int kClusterCtas = 8, kClusterThreads = 256, kClusterChunk = kClusterThreads * kScanPer;
constexpr int kClusterBatch = 4;

__device__ __forceinline__ void cells_barrier() {
    __threadfence();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    __threadfence();
}

__global__ void __cluster_dims__(kClusterCtas, 1, 1) __launch_bounds__(kClusterThreads)
    cells_rebuild_kernel(const double *__restrict__ x, int n, CellList c, unsigned long long *list_n, double *xref,
                         const int *vl, int *err) {
    if ((*vl & 1) == 0) return;   // (uniform over the cluster; vl is the check kernel's)
    __shared__ int s_warp[33];
    const int tid = threadIdx.x, gt = blockIdx.x * kClusterThreads + tid, stride = kClusterCtas * kClusterThreads;
    constexpr int B = kClusterBatch;
    for (int i0 = gt; i0 < n; i0 += B * stride) {
        double p[B][3];
#pragma unroll
        for (int k = 0; k < B; ++k)
            if (i0 + k * stride < n)
                for (int d = 0; d < 3; ++d) p[k][d] = x[3 * static_cast<size_t>(i0 + k * stride) + d];
#pragma unroll
        for (int k = 0; k < B; ++k) {
            const int i = i0 + k * stride;
            if (i >= n) break;
            for (int d = 0; d < 3; ++d) xref[3 * static_cast<size_t>(i) + d] = p[k][d];
            bin_particle(c, i, p[k][0], p[k][1], p[k][2]);
        }
    }
    if (gt == 0) *list_n = 0;
    cells_barrier();
    const int nch = (c.H + kClusterChunk - 1) / kClusterChunk;
    for (int ch = blockIdx.x; ch < nch; ch += kClusterCtas) {   // scan within each chunk
        const int base = ch * kClusterChunk + tid * kScanPer;
        int v[kScanPer];
        scan_load(c.cnt, base, c.H, v);
        const int total = block_exclusive_scan<kClusterThreads>(v, s_warp);
        scan_store(c.start, base, c.H, v);
        if (tid == 0) {
            c.bsum[ch] = total;
            if (ch == nch - 1) c.start[c.H] = n;   // every particle is in one bucket
        }
    }
    cells_barrier();
    if (nch > 1) {
        for (int ch = blockIdx.x; ch < nch; ch += kClusterCtas) {   // ... and the chunks before it
            const int base = ch * kClusterChunk + tid * kScanPer;
            int sum = 0, v[kScanPer];
            scan_load(c.start, base, c.H, v);
            for (int k = 0; k < ch; ++k) sum += c.bsum[k];
            for (int k = 0; k < kScanPer; ++k) v[k] += sum;
            scan_store(c.start, base, c.H, v);
        }
        cells_barrier();
    }
    for (int i0 = gt; i0 < n; i0 += B * stride) {   // scatter_particle, B at a time
        uint32_t key[B];
        int s0[B], s1[B], at[B];
#pragma unroll
        for (int k = 0; k < B; ++k) key[k] = i0 + k * stride < n ? c.key[i0 + k * stride] : 0u;
#pragma unroll
        for (int k = 0; k < B; ++k) {
            s0[k] = c.start[key[k]];
            s1[k] = c.start[key[k] + 1];
            at[k] = i0 + k * stride < n ? atomicSub(&c.cnt[key[k]], 1) - 1 : 0;
        }
#pragma unroll
        for (int k = 0; k < B; ++k) {
            const int i = i0 + k * stride, pos = s0[k] + at[k];
            if (i >= n) break;
            if (pos >= s0[k] && pos < s1[k])
                c.sorted[pos] = i;
            else
                atomicOr(err, DEV_ERR_BOUNDS);
        }
    }
    cells_barrier();
    for (int b0 = gt; b0 < c.H; b0 += B * stride) {   // sort_bucket, the pairs (nearly all there is to sort) B at a time
        int s0[B], m[B], u[B], v[B];
#pragma unroll
        for (int k = 0; k < B; ++k) {
            const int b = b0 + k * stride;
            s0[k] = b < c.H ? c.start[b] : 0;
            m[k] = b < c.H ? c.start[b + 1] - s0[k] : 0;
        }
#pragma unroll
        for (int k = 0; k < B; ++k)
            if (m[k] == 2) {
                u[k] = c.sorted[s0[k]];
                v[k] = c.sorted[s0[k] + 1];
            }
#pragma unroll
        for (int k = 0; k < B; ++k) {
            if (m[k] == 2 && u[k] > v[k]) {
                c.sorted[s0[k]] = v[k];
                c.sorted[s0[k] + 1] = u[k];
            }
            if (m[k] > 2) sort_bucket(c.start, c.sorted, b0 + k * stride);
        }
    }
}

cudaError_t launch_rebuild_cells(sd_handle *h, cudaStream_t st, const double *x64) {
    cells_rebuild_kernel<<<kClusterCtas, kClusterThreads, 0, st>>>(x64, h->n, h->cl, h->vn, h->xref, h->d_vl, h->d_err);
    ++h->launches;
    return cudaGetLastError();
}

// ---------------------------------------------------------------- forces (Sec. 3.1, step 2)

// F_i = F_ext,i + g + sum_{j: r_ij < r_c} 12 eps (2a)^12 r^-14 (r_i - r_j)
// (U = eps (2a/r)^12, truncated at r_c, F = -grad U; Sec. 3.1 step 2), and with
// lubrication (vlag != nullptr) the singular friction of Sec. 2.3 Eq. lubrication,
//   F_i -= (1/mu0) sum_{j: 0 < s < 1} [(1/(4s) - (9/40) ln s) e e^T - (1/6) ln s (I - e e^T)] (v_i - v_j),
// s = r/a - 2, e = r_ij / r, with the previous step's velocities vlag (Sec. 3.1:
// the forces are corrected for lubrication before the velocity update).  FP64;
// writes F64 and its mirror.
template <typename V4>
__global__ void forces_rep_kernel(const double *__restrict__ x, const double *__restrict__ fext, double gx, double gy,
                                  double gz, double eps, double rc, double s12, const double *__restrict__ vlag,
                                  double inv_a, double inv_mu0, CellList c, int n, int npad, double *__restrict__ F,
                                  V4 *__restrict__ m, float *__restrict__ soa, int *err) {
    // kWalkLanes threads per particle, partial sums meet in a fixed shuffle tree
    const long long gt = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int i = static_cast<int>(gt / kWalkLanes), sub = static_cast<int>(gt % kWalkLanes);
    const bool active = i < n;
    const bool rep = eps != 0.0, lub = vlag != nullptr;
    const double rc2 = rep ? rc * rc : 0.0;
    const double rl2 = lub ? 9.0 / (inv_a * inv_a) : 0.0;   // (3a)^2
    const double rmax2 = rc2 > rl2 ? rc2 : rl2;
    double f[3] = {0.0, 0.0, 0.0};
    bool coincident = false, found = false;
    if (active) {
        const double xi = x[3 * i], yi = x[3 * i + 1], zi = x[3 * i + 2];
        for_each_neighbour_part(c, i, c.cell[i], sub, kWalkLanes, [&](int j) {
            double dx = xi - x[3 * j], dy = yi - x[3 * j + 1], dz = zi - x[3 * j + 2];
            box_image(c.box, dx, dy, dz);
            const double r2 = dx * dx + dy * dy + dz * dz;
            if (r2 >= rmax2) return;
            found = true;
            if (r2 == 0.0) {
                if (rep) coincident = true;   // s = -2: no lubrication term
                return;
            }
            const double ri = rsqrt_nr64(r2);   // no FP64 division (scarce FP64 throughput)
            if (r2 < rc2) {
                const double ir2 = ri * ri;
                const double ir6 = ir2 * ir2 * ir2;
                const double coef = 12.0 * eps * s12 * ir6 * ir6 * ir2;
                f[0] += coef * dx;
                f[1] += coef * dy;
                f[2] += coef * dz;
            }
            if (lub) {
                // the gap s in FP64 (it cancels: r/a - 2); the coefficients in the
                // working precision of the pair terms (FP32 in the FP32 modes)
                const double sg = r2 * ri * inv_a - 2.0;
                if (sg > 0.0 && sg < 1.0) {
                    double zn, zt;
                    if constexpr (std::is_same<V4, float4>::value) {
                        const float sf = static_cast<float>(sg), ls = logf(sf);
                        zn = __fsub_rn(__fdiv_rn(0.25f, sf), __fmul_rn(0.225f, ls));
                        zt = __fmul_rn(ls, -1.0f / 6.0f);
                    } else {
                        const double ls = log(sg);
                        zn = 0.25 / sg - 0.225 * ls;
                        zt = -ls / 6.0;
                    }
                    const double ex = dx * ri, ey = dy * ri, ez = dz * ri;
                    const double wx = vlag[3 * i] - vlag[3 * j], wy = vlag[3 * i + 1] - vlag[3 * j + 1],
                                 wz = vlag[3 * i + 2] - vlag[3 * j + 2];
                    const double en = ex * wx + ey * wy + ez * wz;
                    // zeta w = zn (e.w) e + zt (w - (e.w) e)
                    const double kn = (zn - zt) * en;
                    f[0] -= inv_mu0 * (kn * ex + zt * wx);
                    f[1] -= inv_mu0 * (kn * ey + zt * wy);
                    f[2] -= inv_mu0 * (kn * ez + zt * wz);
                }
            }
        });
    }
    const int writer = walk_combine(f, found, sub);
    coincident = walk_any(coincident);
    if (!active || sub != writer) return;
    const double f0 = f[0] + fext[3 * i] + gx, f1 = f[1] + fext[3 * i + 1] + gy, f2v = f[2] + fext[3 * i + 2] + gz;
    if (coincident) atomicOr(err, DEV_ERR_COINCIDENT);
    if (!isfinite(f0) || !isfinite(f1) || !isfinite(f2v)) atomicOr(err, DEV_ERR_NONFINITE);
    F[3 * i] = f0;
    F[3 * i + 1] = f1;
    F[3 * i + 2] = f2v;
    put_mirror(m, soa, npad, i, f0, f1, f2v);
}

// Forces of a Verlet step (Sec. 3.1, step 2) with soft repulsion and/or lubrication:
// the pairs come from the steps' near-pair list (it holds every pair within the
// largest cutoff while the list is valid), in FP64; the terms are forces_rep_kernel's.  Plus
// F_ext and gravity.  Writes F64 and the force mirror.
// Some 60 FP64 operations a pair, two a clock and SM, so what counts is that every SM and
// every lane has pairs: in CTAs of 64, L lanes take a particle's run in turn, and its terms
// are added in ascending partner order (entries beyond the cutoff add zeros wherever they
// stand in the run).  One thread per particle in CTAs of 128 left most SMs idle at small n
// (N = 4,913, lubrication: 19 us, with four lanes 13; cold caches); from kForceWideN particles
// on one lane each fills them, and four cost more in the ordered sum.  A step with one lane / four:
// repulsion at phi = 0.1, N = 8,193 77.4 / 74.7 us, 10,240 98.4 / 96.3, 13,824 142.6 / 141.7, 17,408
// 204.9 / 205.2; lubrication on a lattice 83.7 / 81.6, 104.9 / 104.5, 147.6 / 149.2, 210.9 / 217.5.
// The line stands where lubrication's sides meet; both forms give the same bits.
constexpr int kForceWideN = 10752;
template <typename V4, int L>
__global__ void __launch_bounds__(64) forces_list_kernel(const double *__restrict__ x, const double *__restrict__ fext, double gx,
                                   double gy, double gz, double eps, double rc, double s12,
                                   const double *__restrict__ vlag, double inv_a, double inv_mu0, CellList c,
                                   const int2 *__restrict__ ent, const int *__restrict__ noff,
                                   const int *__restrict__ ncnt, int cap, int n, int npad, double *__restrict__ F,
                                   V4 *__restrict__ m, float *__restrict__ soa, int *err) {
    const long long gt = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int i = static_cast<int>(gt / L), sub = static_cast<int>(gt % L);
    const bool active = i < n;
    const bool rep = eps != 0.0, lub = vlag != nullptr;
    const double rc2 = rep ? rc * rc : 0.0;
    const double rl2 = lub ? 9.0 / (inv_a * inv_a) : 0.0;   // (3a)^2
    const double rmax2 = rc2 > rl2 ? rc2 : rl2;
    double xi = 0.0, yi = 0.0, zi = 0.0;
    if (active) {
        xi = x[3 * i];
        yi = x[3 * i + 1];
        zi = x[3 * i + 2];
    }
    double f[3] = {0.0, 0.0, 0.0};
    bool coincident = false;
    auto pair = [&](int j) {
        double dx = xi - x[3 * j], dy = yi - x[3 * j + 1], dz = zi - x[3 * j + 2];
        box_image(c.box, dx, dy, dz);
        const double r2 = dx * dx + dy * dy + dz * dz;
        if (r2 >= rmax2) return;
        if (r2 == 0.0) {
            if (rep) coincident = true;   // s = -2: no lubrication term
            return;
        }
        const double ri = rsqrt_nr64(r2);
        if (r2 < rc2) {
            const double ir2 = ri * ri;
            const double ir6 = ir2 * ir2 * ir2;
            const double coef = 12.0 * eps * s12 * ir6 * ir6 * ir2;
            f[0] += coef * dx;
            f[1] += coef * dy;
            f[2] += coef * dz;
        }
        if (lub) {
            const double sg = r2 * ri * inv_a - 2.0;
            if (sg > 0.0 && sg < 1.0) {
                double zn, zt;
                if constexpr (std::is_same<V4, float4>::value) {
                    const float sf = static_cast<float>(sg), ls = logf(sf);
                    zn = __fsub_rn(__fdiv_rn(0.25f, sf), __fmul_rn(0.225f, ls));
                    zt = __fmul_rn(ls, -1.0f / 6.0f);
                } else {
                    const double ls = log(sg);
                    zn = 0.25 / sg - 0.225 * ls;
                    zt = -ls / 6.0;
                }
                const double ex = dx * ri, ey = dy * ri, ez = dz * ri;
                const double wx = vlag[3 * i] - vlag[3 * j], wy = vlag[3 * i + 1] - vlag[3 * j + 1],
                             wz = vlag[3 * i + 2] - vlag[3 * j + 2];
                const double en = ex * wx + ey * wy + ez * wz;
                const double kn = (zn - zt) * en;
                f[0] -= inv_mu0 * (kn * ex + zt * wx);
                f[1] -= inv_mu0 * (kn * ey + zt * wy);
                f[2] -= inv_mu0 * (kn * ez + zt * wz);
            }
        }
    };
    const int cnt = active ? ncnt[i] : 0;
    double sum[3] = {0.0, 0.0, 0.0};
    if (cnt < 0) {   // a particle the overflowed list corrects in place: the cell list (rebuilt
                     // every step while the list overflows) gives its pairs
        for_each_neighbour_part(c, i, c.cell[i], sub, L, pair);
    }
    if (__any_sync(0xffffffffu, cnt < 0))
#pragma unroll
        for (int l = 0; l < L; ++l)
            for (int d = 0; d < 3; ++d) sum[d] += __shfl_sync(0xffffffffu, cnt < 0 ? f[d] : 0.0, l, L);
    const long long e0 = cnt > 0 ? dbg_index(noff[i], static_cast<long long>(cap) - cnt + 1, err) : 0;
    const int rounds = __reduce_max_sync(0xffffffffu, (max(cnt, 0) + L - 1) / L);
    for (int r = 0; r < rounds; ++r) {
        const int k = r * L + sub;
        f[0] = f[1] = f[2] = 0.0;
        if (k < cnt) pair(static_cast<int>(dbg_index(ent[e0 + k].y, n, err)));
#pragma unroll
        for (int l = 0; l < L; ++l)
            for (int d = 0; d < 3; ++d) sum[d] += __shfl_sync(0xffffffffu, f[d], l, L);
    }
    coincident = __any_sync(0xffffffffu, coincident);
    if (!active || sub != 0) return;
    const double f0 = sum[0] + fext[3 * i] + gx, f1 = sum[1] + fext[3 * i + 1] + gy, f2v = sum[2] + fext[3 * i + 2] + gz;
    if (coincident) atomicOr(err, DEV_ERR_COINCIDENT);
    if (!isfinite(f0) || !isfinite(f1) || !isfinite(f2v)) atomicOr(err, DEV_ERR_NONFINITE);
    F[3 * i] = f0;
    F[3 * i + 1] = f1;
    F[3 * i + 2] = f2v;
    put_mirror(m, soa, npad, i, f0, f1, f2v);
}

cudaError_t launch_forces_list(sd_handle *h, cudaStream_t st, const double *x64) {
    if (h->n == 0) return cudaSuccess;
    const bool wide = h->n < kForceWideN;
    const int nb = static_cast<int>((static_cast<long long>(h->n) * (wide ? 4 : 1) + 63) / 64);
    const double *g = h->cfg.gravity;
    const double s12 = pow(2.0 * h->cfg.a, 12.0);
    const double *vlag = h->lub ? h->vlag : nullptr;
    const double inv_a = 1.0 / h->pc.a, inv_mu0 = 1.0 / h->pc.mu0;
    prof_begin(h, SD_KERNEL_FORCES, st);
#define SD_FORCES(VV, LL)                                                                                            \
    forces_list_kernel<VV, LL><<<nb, 64, 0, st>>>(x64, h->fext64, g[0], g[1], g[2], h->cfg.rep_eps, h->rep_rc, s12, vlag, \
                                                  inv_a, inv_mu0, h->cl, h->vent, h->voff, h->vcnt, h->near_cap, h->n,   \
                                                  h->npad, h->F64, static_cast<VV *>(h->frcm.aos), h->frcm.soa, h->d_err)
    if (h->mode == MODE_FP64) {
        if (wide) SD_FORCES(dbl4, 4); else SD_FORCES(dbl4, 1);
    } else {
        if (wide) SD_FORCES(float4, 4); else SD_FORCES(float4, 1);
    }
#undef SD_FORCES
    prof_end(h, SD_KERNEL_FORCES, st);
    ++h->launches;
    return cudaGetLastError();
}

cudaError_t launch_forces_rep(sd_handle *h, cudaStream_t st, const double *x64) {
    if (h->n == 0) return cudaSuccess;
    const int nb = static_cast<int>((static_cast<long long>(h->n) * kWalkLanes + 127) / 128);
    const double *g = h->cfg.gravity;
    const double s12 = pow(2.0 * h->cfg.a, 12.0);
    prof_begin(h, SD_KERNEL_FORCES, st);
    const double *vlag = h->lub ? h->vlag : nullptr;
    const double inv_a = 1.0 / h->pc.a, inv_mu0 = 1.0 / h->pc.mu0;
    if (h->mode == MODE_FP64)
        forces_rep_kernel<dbl4><<<nb, 128, 0, st>>>(x64, h->fext64, g[0], g[1], g[2], h->cfg.rep_eps, h->rep_rc, s12,
                                                    vlag, inv_a, inv_mu0, h->cl, h->n, h->npad, h->F64,
                                                    static_cast<dbl4 *>(h->frcm.aos), h->frcm.soa, h->d_err);
    else
        forces_rep_kernel<float4><<<nb, 128, 0, st>>>(x64, h->fext64, g[0], g[1], g[2], h->cfg.rep_eps, h->rep_rc,
                                                      s12, vlag, inv_a, inv_mu0, h->cl, h->n, h->npad, h->F64,
                                                      static_cast<float4 *>(h->frcm.aos), h->frcm.soa, h->d_err);
    prof_end(h, SD_KERNEL_FORCES, st);
    ++h->launches;
    return cudaGetLastError();
}

}  // namespace sd
