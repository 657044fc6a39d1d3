// neighbours.cuh -- walk over the hashed cell list (built in cells.cu).
#pragma once
#include "sd_internal.h"

namespace sd {

// A neighbour cell coordinate: wrapped in a periodic dimension (nc > 0).
__device__ __forceinline__ int cell_wrap(int c, int nc) {
    if (nc <= 0) return c;
    return c < 0 ? c + nc : (c >= nc ? c - nc : c);
}

// Calls f(j) for every particle j != i in one of the 27 cells around cell ci, in fixed order
// (cells by offset, bucket entries by index), split over `step` cooperating threads: this
// thread visits the cells first, first + step, ...
template <typename Fn>
__device__ __forceinline__ void for_each_neighbour_part(const CellList &c, int i, int4 ci, int first, int step,
                                                        Fn &&f) {
    for (int k = first; k < 27; k += step) {
        const int cx = cell_wrap(ci.x + (k % 3) - 1, c.nc[0]), cy = cell_wrap(ci.y + (k / 3) % 3 - 1, c.nc[1]),
                  cz = cell_wrap(ci.z + k / 9 - 1, c.nc[2]);
        const uint32_t b = cell_hash(cx, cy, cz, c.H);
        const int s1 = c.start[b + 1];
        for (int s = c.start[b]; s < s1; ++s) {
            const int j = static_cast<int>(dbg_index(c.sorted[dbg_index(s, c.n, c.err)], c.n, c.err));
            if (j == i) continue;
            const int4 cj = c.cell[j];
            if (cj.x != cx || cj.y != cy || cj.z != cz) continue;
            f(j);
        }
    }
}

// ---------------------------------------------------------------- mirrors and bins

// Entry i of a mirror: (x, y, z, 0) in the AoS array and, if present, the SoA copy.
template <typename V4>
__device__ __forceinline__ void put_mirror(V4 *aos, float *soa, int npad, int i, double x, double y, double z) {
    V4 v;
    v.x = x;
    v.y = y;
    v.z = z;
    v.w = 0;
    aos[i] = v;
    if (soa) {
        soa[i] = static_cast<float>(x);
        soa[npad + i] = static_cast<float>(y);
        soa[2 * static_cast<size_t>(npad) + i] = static_cast<float>(z);
    }
}

// u wrapped into [0, L) in a periodic dimension (L > 0), unchanged otherwise.
__device__ __forceinline__ double wrap_box(double u, double L, double invL) {
    return L > 0.0 ? u - L * floor(u * invL) : u;
}

// Mirror entry of a position: relative to particle 0 (only differences enter the
// pair terms, and small coordinates keep FP32 separations accurate), wrapped into
// the box in periodic dimensions (the pair terms take the nearest image).
template <typename V4>
__device__ __forceinline__ void put_pos_mirror(V4 *m, float *soa, int npad, int i, const double *x, const Box &b) {
    const double px = x[3 * i], py = x[3 * i + 1], pz = x[3 * i + 2];
    put_mirror(m, soa, npad, i, wrap_box(px - x[0], b.L[0], b.invL[0]), wrap_box(py - x[1], b.L[1], b.invL[1]),
               wrap_box(pz - x[2], b.L[2], b.invL[2]));
}

// (the conversion rounds down and saturates by itself: two FP64-rate operations instead of five,
// which is what a build on a few SMs waits for; then the range is kept for absurd coordinates)
__device__ __forceinline__ int cell_coord(double x, double inv_h) {
    return min(max(__double2int_rd(x * inv_h), -1000000000), 1000000000);
}

// Cell coordinate in dimension d: nc[d] cells over [0, L) of the wrapped coordinate
// in a periodic dimension, cells of side h otherwise.
__device__ __forceinline__ int cell_coord_d(const CellList &c, int d, double x) {
    const int nc = c.nc[d];
    if (nc <= 0) return cell_coord(x, c.inv_h);
    const int k = __double2int_rd(wrap_box(x, c.box.L[d], c.box.invL[d]) * c.box.invL[d] * nc);
    return k < 0 ? 0 : (k >= nc ? nc - 1 : k);
}

// Particle i's cell and bucket; counts it there.
__device__ __forceinline__ void bin_particle(const CellList &c, int i, double px, double py, double pz) {
    const int cx = cell_coord_d(c, 0, px);
    const int cy = cell_coord_d(c, 1, py);
    const int cz = cell_coord_d(c, 2, pz);
    c.cell[i] = make_int4(cx, cy, cz, 0);
    const uint32_t k = cell_hash(cx, cy, cz, c.H);
    c.key[i] = k;
    atomicAdd(&c.cnt[k], 1);
}

constexpr int kScanPer = 16;   // buckets a thread scans (both arrays are aligned to 64 bytes and hold whole
                               // groups of them, 1,024 or a larger power of two: four 16-byte accesses)
__device__ __forceinline__ void scan_load(const int *in, int base, int H, int (&v)[kScanPer]) {
#pragma unroll
    for (int k = 0; k < kScanPer; k += 4) {
        const int4 q = base < H ? *reinterpret_cast<const int4 *>(in + base + k) : make_int4(0, 0, 0, 0);
        v[k] = q.x; v[k + 1] = q.y; v[k + 2] = q.z; v[k + 3] = q.w;
    }
}
__device__ __forceinline__ void scan_store(int *out, int base, int H, const int (&v)[kScanPer]) {
    if (base >= H) return;
#pragma unroll
    for (int k = 0; k < kScanPer; k += 4)
        *reinterpret_cast<int4 *>(out + base + k) = make_int4(v[k], v[k + 1], v[k + 2], v[k + 3]);
}

// Exclusive scan of kScanPer values per thread across a block; returns the
// block total.  Warp shuffles within warps, shared memory across warps.
template <int NT>
__device__ __forceinline__ int block_exclusive_scan(int v[kScanPer], int *s_warp) {
    int tsum = 0;
    for (int k = 0; k < kScanPer; ++k) {
        const int t = v[k];
        v[k] = tsum;
        tsum += t;
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int incl = tsum;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        int w = (lane < NT / 32) ? s_warp[lane] : 0;
        int wi = w;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        s_warp[lane] = wi - w;  // exclusive warp offsets
        if (lane == 31) s_warp[32] = wi;
    }
    __syncthreads();
    const int off = s_warp[wid] + incl - tsum;
    for (int k = 0; k < kScanPer; ++k) v[k] += off;
    const int total = s_warp[32];
    __syncthreads();
    return total;
}

// Particle i takes a place in its bucket by counting the bucket's occupancy down, which
// leaves every counter at zero for the next build (no memset).
__device__ __forceinline__ void scatter_particle(const uint32_t *key, const int *start, int *cnt, int *sorted, int i,
                                                 int *err) {
    const uint32_t k = key[i];
    const int pos = start[k] + atomicSub(&cnt[k], 1) - 1;
    if (pos >= start[k] && pos < start[k + 1])   // always, unless a counter was left non-zero
        sorted[pos] = i;
    else
        atomicOr(err, DEV_ERR_BOUNDS);
}

// Sort bucket b by particle index (buckets hold ~1 particle; a bucket larger
// than 256 -- only possible for unphysically dense input -- stays unsorted, which
// changes only the FP64 summation order of its near pairs).
__device__ __forceinline__ void sort_bucket(const int *start, int *sorted, int b) {
    const int s0 = start[b], s1 = start[b + 1];
    if (s1 - s0 < 2 || s1 - s0 > 256) return;
    for (int p = s0 + 1; p < s1; ++p) {
        const int v = sorted[p];
        int q = p - 1;
        while (q >= s0 && sorted[q] > v) {
            sorted[q + 1] = sorted[q];
            --q;
        }
        sorted[q + 1] = v;
    }
}

// Nearest-image FP64 separation r_i - r_j (identity in unbounded dimensions).  Most pairs
// need no image: |d| below half a period rounds to zero periods, and a comparison of the upper
// words (integers) says so without the twelve FP64 operations (two a clock and SM).
__device__ __forceinline__ bool within_half(double d, double L) {
    return L == 0.0 || (__double2hiint(d) & 0x7fffffff) < __double2hiint(0.5 * L);
}
__device__ __forceinline__ void box_image(const Box &b, double &dx, double &dy, double &dz) {
    if (!b.periodic) return;
    if (within_half(dx, b.L[0]) && within_half(dy, b.L[1]) && within_half(dz, b.L[2])) return;
    dx = min_image_f64(dx, b.L[0], b.invL[0]);
    dy = min_image_f64(dy, b.L[1], b.invL[1]);
    dz = min_image_f64(dz, b.L[2], b.invL[2]);
}

// Threads per particle in the neighbour-walking kernels (a power of two <= 32;
// consecutive lanes of one warp), and the fixed-order sum over them.
constexpr int kWalkLanes = 8;

__device__ __forceinline__ double walk_sum(double v) {
    for (int o = kWalkLanes / 2; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Lanes of this thread's group whose flag `b` is set (bit k = sub-lane k).
__device__ __forceinline__ unsigned walk_mask(bool b) {
    const unsigned m = __ballot_sync(0xffffffffu, b);
    const int lane = threadIdx.x & 31;
    return (m >> (lane & ~(kWalkLanes - 1))) & ((1u << kWalkLanes) - 1u);
}

// Combine per-lane FP64 partial sums v[0..K) of a group.  Most groups have at
// most one lane with a non-zero contribution (that lane's sums are the result,
// no arithmetic); only when some group in the warp has two or more does the
// warp run the fixed shuffle tree.  Returns the sub-lane that holds the result.
template <int K>
__device__ __forceinline__ int walk_combine(double (&v)[K], bool contributed, int sub) {
    const unsigned gm = walk_mask(contributed);
    const bool many = __popc(gm) > 1;
    if (__any_sync(0xffffffffu, many)) {
        for (int d = 0; d < K; ++d) v[d] = walk_sum(v[d]);
        return 0;
    }
    (void)sub;
    return gm ? __ffs(gm) - 1 : 0;
}
__device__ __forceinline__ bool walk_any(bool b) {
    const unsigned m = __ballot_sync(0xffffffffu, b);
    const int lane = threadIdx.x & 31;
    const unsigned grp = ((1u << kWalkLanes) - 1u) << (lane & ~(kWalkLanes - 1));
    return (m & grp) != 0u;
}

}  // namespace sd
