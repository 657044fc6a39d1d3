// small.cu -- one launch for the whole product, or for many Euler steps, of a small
// system with constant forces (Sec. 3.1, steps 1 and 3).
//
// What bounds a small system is not arithmetic but the chain of launches of a step
// (check, list rebuild, near pass, all-pairs kernel, epilogue) and of dependent loads and
// FP64 operations in each: N = 1,021 has 0.6 us of FP32 work per step on the whole chip
// and took 25 us through those kernels, four spheres in FP64 80 us, set_positions and one
// product at N = 1,000 106 us.  Through this one: 6.8 us, 2.6 us and 24 us (about half of
// it the host's two calls).
// Here a step is two phases of one kernel:
//   A  a thread-block cluster takes a block of targets, its CTAs the j-splits; each sums
//      the block over its sources and hands every row's sum to the CTA of the cluster
//      that updates the row, through distributed shared memory;
//   B  the splits' sums of a row are added in ascending order, the self term joins, and v
//      or x + dt v is written;
// with a hardware cluster barrier between the two.  Between steps the CTAs exchange
// positions without a grid barrier: every 8-byte word of an exchanged position carries
// four bytes of it and the step's number, so a reader polls (bounded) the words it needs
// until they are of its step (one write and one read of latency, where a barrier and the
// loads after it cost twice that).  Two exchange buffers in turn are enough: a row of step
// k + 2 is written only after its cluster has read every row of step k + 1, and each of
// those was written after its own cluster had read all of step k.  The launch is
// cooperative, so all CTAs are resident; a single product exchanges nothing.
// The state is FP64 and each step starts from its positions relative to its particle 0,
// so a step is a pure function of the state: any split of a trajectory into launches gives
// the same bits.  A system that fits one CTA keeps its positions in shared memory.
//   FP32C: packed pair terms (two sources per instruction) with r^2 clamped to (2a)^2,
//     folded into (hi, lo) sums; the pairs within 1.01 r_near are noted as they are met
//     (a test of r^2 that the pair term needs anyway), and each noted pair closer than
//     r_near adds the exact FP64 term minus the clamped FP32 one: no cell list and no
//     neighbour list.  The FP64 terms are a chain of some 20 dependent FP64 operations
//     (about 2,500 cycles), so an extra warp evaluates the last step's pairs at the new
//     positions while the others run the loop; what is new is evaluated after it.  The
//     noted pairs are ranked by (target, source) before they are summed, so the result
//     depends neither on the order of notes nor on what was noted before.
//   FP64: the pair term in FP64; pairs closer than 2a (the self pair among them) leave
//     the common path, so no clamp and no near pass are needed.
#include <algorithm>
#include <type_traits>
#include "sd_internal.h"

namespace sd {

constexpr int kSmWarps = 16;               // one CTA per SM; 16 warps share a block of targets
constexpr int kSmThreads = 32 * kSmWarps + 32;   // ... and one more takes the near pairs of the last step
constexpr int kSmAhead = 64;               // near pairs evaluated ahead (more: after the loop, by all threads)
constexpr int kSmNotes = 512;              // noted pairs a CTA holds; more: its targets scan their range again
constexpr double kSmDense = 8192.0;        // expected near pairs (known in a box) from which the near pass's full warps
                                           // win: an fcc lattice of 2,048 52 us a step here, 35 there; 864: 29 and 41
constexpr int kSmSoloFP32 = 128;           // largest n one CTA takes (FP32C)
constexpr int kSmSoloFP64 = 16;            // ... FP64: two FP64 operations a clock and SM, so more SMs sooner
constexpr int kSmMaxSteps = 512;           // steps per launch
constexpr int kSmMaxSplit = 8;             // (the portable cluster size)

struct SmallArgs {
    double *x0, *x1;          // step k reads x_k and writes x_{k+1}: x0 / x1 in turn, or
    size_t stride;            // (stride > 0) x0 + k stride
    const void *F;            // n x 3 forces
    int f32;                  // ... float (1) or double (0)
    void *vout;               // velocities of rows row0 .. row1-1 (OUT_F32, OUT_F64)
    int out;                  // OUT_F32, OUT_F64 or OUT_EULER
    int n, nsplit, jlen;      // j-splits (= CTAs per cluster), sources per split (a multiple of 4)
    int rows, lnt;            // rows of a block that one CTA of the cluster updates; log2 of the CTA's targets
    int nbl, wb, iw, span;    // target blocks per CTA (solo: all), warps per block; FP64: targets per warp, lanes in use (powers of two <= 32)
    int nsteps, solo, row0, row1;
    double dt, rnear2;
    float rscreen2;
    PairConst pc;
    PairConst2 c2;
    ulonglong2 *xch;          // [2][3 n] exchanged positions: (low half, tag), (high half, tag)
    unsigned *sync;           // [0] tag of the launch's first exchanged step, [1] a wait ran out, [2] CTAs done
    int *err;
    long long wd;
};

__device__ __forceinline__ double wrap_coord(double u, double L, double invL) {
    return L > 0.0 ? u - L * floor(u * invL) : u;
}

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address in CTA `rank` of the cluster of *p (in this CTA's shared memory), and a
// store to such an address.
__device__ __forceinline__ uint32_t cluster_addr(const void *p, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_store(uint32_t p, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(p), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_store(uint32_t p, int v) {
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(p), "r"(v) : "memory");
}

// Write / read (polling, bounded) one exchanged FP64 value of the step `tag`.
__device__ __forceinline__ void xch_put(ulonglong2 *p, double v, unsigned tag) {
    const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(v));
    const unsigned long long t = static_cast<unsigned long long>(tag) << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"((b & 0xffffffffull) | t),
                 "l"((b >> 32) | t)
                 : "memory");
}
__device__ __forceinline__ bool xch_ready(const ulonglong2 &w, unsigned tag) {
    return static_cast<unsigned>(w.x >> 32) == tag && static_cast<unsigned>(w.y >> 32) == tag;
}
__device__ __forceinline__ ulonglong2 xch_load(const ulonglong2 *p) {
    ulonglong2 w;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w.x), "=l"(w.y) : "l"(p) : "memory");
    return w;
}
__device__ __forceinline__ double xch_value(const ulonglong2 &w) {
    return __longlong_as_double(static_cast<long long>((w.x & 0xffffffffull) | (w.y << 32)));
}
// The coordinates of the particles 0 and p (polled together: one round trip); false once
// the wait has run out here or elsewhere.
__device__ __forceinline__ bool xch_get(const SmallArgs &a, const ulonglong2 *buf, int p, unsigned tag, double (&o)[3],
                                        double (&v)[3]) {
    const ulonglong2 *q = buf + 3 * static_cast<size_t>(p);
    bool ok = false;
    for (long long it = 0; it < a.wd; ++it) {
        ulonglong2 w[6];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            w[d] = xch_load(buf + d);
            w[3 + d] = xch_load(q + d);
        }
        ok = true;
#pragma unroll
        for (int d = 0; d < 6; ++d) ok = ok && xch_ready(w[d], tag);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            o[d] = xch_value(w[d]);
            v[d] = xch_value(w[3 + d]);
        }
        if (ok) break;
        if ((it & 63) == 63 && *reinterpret_cast<volatile unsigned *>(a.sync + 1)) break;
    }
    if (!ok) {
        atomicOr(a.err, DEV_ERR_TIMEOUT);
        *reinterpret_cast<volatile unsigned *>(a.sync + 1) = 1u;
    }
    return ok;
}

// What a CTA's near pairs are evaluated from: its sources and targets in shared memory.
struct SmallNear {
    const float *src, *tgt;   // [6][jlen], [3][nt]
    const double *pd;         // [3][jlen + nt]
    int jlen, nt, j0;
};
// The noted pair `key` = (target << 16 | source): the exact FP64 term minus the clamped
// FP32 one the loop added, if r < r_near (the near pass of epilogue.cu for one pair).  Out
// of line: the step's code is fetched anew every step, and one copy serves three callers.
template <int TENSOR, bool PER>
__device__ __noinline__ bool small_near(const SmallArgs &a, const SmallNear &m, int key, double *c) {
    constexpr int TD = (TENSOR == T_OSEEN) ? T_OSEEN : T_RP;
    const int t = static_cast<int>(dbg_index(key >> 16, m.nt, a.err)),
              q = static_cast<int>(dbg_index(key & 0xffff, m.jlen, a.err)), pd = m.jlen + m.nt, u = m.jlen + t;
    double dx = m.pd[u] - m.pd[q], dy = m.pd[pd + u] - m.pd[pd + q], dz = m.pd[2 * pd + u] - m.pd[2 * pd + q];
    if (PER) {
        dx = min_image_f64(dx, a.pc.Ld[0], a.pc.invLd[0]);
        dy = min_image_f64(dy, a.pc.Ld[1], a.pc.invLd[1]);
        dz = min_image_f64(dz, a.pc.Ld[2], a.pc.invLd[2]);
    }
    const double r2 = dx * dx + dy * dy + dz * dz;
    c[0] = c[1] = c[2] = 0.0;
    if (!(r2 < a.rnear2)) return false;
    if (r2 == 0.0 && TENSOR != T_RPY) {
        atomicOr(a.err, DEV_ERR_COINCIDENT);
        return false;
    }
    double f[3];
    for (int d = 0; d < 3; ++d) {
        const size_t k = 3 * static_cast<size_t>(m.j0 + q) + d;
        f[d] = a.f32 ? static_cast<double>(static_cast<const float *>(a.F)[k]) : static_cast<const double *>(a.F)[k];
    }
    double A, B, dA, dB;
    profile_exact<TENSOR>(r2, a.pc, A, B, dA, dB);
    const double s = B * (dx * f[0] + dy * f[1] + dz * f[2]);
    const int jl = m.jlen;
    float tx = 0.0f, ty = 0.0f, tz = 0.0f;
    pair_f32<TD, true, PER>(m.tgt[t], m.tgt[m.nt + t], m.tgt[2 * m.nt + t],
                            make_float4(m.src[q], m.src[jl + q], m.src[2 * jl + q], 0.0f),
                            make_float4(m.src[3 * jl + q], m.src[4 * jl + q], m.src[5 * jl + q], 0.0f), a.pc, tx, ty, tz);
    c[0] = A * f[0] + s * dx - static_cast<double>(tx);
    c[1] = A * f[1] + s * dy - static_cast<double>(ty);
    c[2] = A * f[2] + s * dz - static_cast<double>(tz);
    return true;
}

// One pair of the FP64 sum, divided by c1 (phase B multiplies the sums).  Closer than 2a: the
// self pair adds nothing (its term mu_ii / mu0 = I joins in phase B), an overlapping pair its
// exact term.  25 FP64 operations, no conversions and no FP64 comparison: they bound the
// larger systems (two a clock and SM), and their chain the smallest
// (with them the product at n = 1,000 75 us, 512 steps of four spheres 1.39 ms; now 63 and 1.31).
template <int TENSOR, bool PER>
__device__ __forceinline__ void small_pair64(double xi, double yi, double zi, double px, double py, double pz, double fx,
                                             double fy, double fz, bool self, const SmallArgs &a, double &ax,
                                             double &ay, double &az) {
    double dx = __dsub_rn(xi, px), dy = __dsub_rn(yi, py), dz = __dsub_rn(zi, pz);
    if (PER) {
        dx = min_image_f64(dx, a.pc.Ld[0], a.pc.invLd[0]);
        dy = min_image_f64(dy, a.pc.Ld[1], a.pc.invLd[1]);
        dz = min_image_f64(dz, a.pc.Ld[2], a.pc.invLd[2]);
    }
    const double r2 = __fma_rn(dz, dz, __fma_rn(dy, dy, __dmul_rn(dx, dx)));
    double A, B;
    if (less_pos64(r2, a.pc.r2min_d)) {
        if (self) return;
        if (r2 == 0.0 && TENSOR != T_RPY) {
            atomicOr(a.err, DEV_ERR_COINCIDENT);
            return;
        }
        double dA, dB;
        profile_exact<TENSOR>(r2, a.pc, A, B, dA, dB);
        A *= a.pc.invc1_d;
        B *= a.pc.invc1_d;
    } else {
        profile64<TENSOR>(r2, a.pc, A, B);
    }
    const double s = __dmul_rn(B, __fma_rn(dz, fz, __fma_rn(dy, fy, __dmul_rn(dx, fx))));
    ax = __fma_rn(s, dx, __fma_rn(A, fx, ax));
    ay = __fma_rn(s, dy, __fma_rn(A, fy, ay));
    az = __fma_rn(s, dz, __fma_rn(A, fz, az));
}

template <int MODE, int R>
__host__ __device__ constexpr int small_block() { return MODE == MODE_FP64 ? 32 : 32 * R; }

// Shared memory, in doubles (8-byte parts first): the splits' sums of the rows this CTA
// updates [nsplit][3][rows], the block's sums [3][nt], FP32C: the near corrections
// [kSmNotes][3], those evaluated ahead [kSmAhead][3], the FP64 positions of the sources
// and targets [3][jlen + nt], the notes of two steps and the sorted targets
// [3][kSmNotes] int; solo: the FP64 positions [3 n].  Then 16-byte aligned: sources
// [6][jlen] (x y z Fx Fy Fz), targets [3][nt], the warps' sums [wb][6 or 3][nt], in float
// (FP32C) or double.
__host__ __device__ inline size_t small_words(int mode, int jlen, int nt, int solo, int n) {
    size_t w = 3 * static_cast<size_t>(nt + kSmMaxSplit) + 3 * static_cast<size_t>(nt);
    if (mode != MODE_FP64) w += 3 * (kSmNotes + kSmAhead) + 3 * static_cast<size_t>(jlen + nt) + 3 * kSmNotes / 2;
    if (solo) w += 3 * static_cast<size_t>(n);
    return (w + 1) & ~static_cast<size_t>(1);
}
static size_t small_smem(int mode, int R, int jlen, int nbl, int wb, int solo, int n) {
    const size_t es = mode == MODE_FP64 ? sizeof(double) : sizeof(float);
    const int nt = nbl * (mode == MODE_FP64 ? 32 : 32 * R);
    return sizeof(double) * small_words(mode, jlen, nt, solo, n) +
           es * (6 * static_cast<size_t>(jlen) + 3 * static_cast<size_t>(nt) +
                 static_cast<size_t>(wb) * (mode == MODE_FP64 ? 3 : 6) * nt);
}

template <int TENSOR, int MODE, bool PER, int R>
__global__ void __launch_bounds__(kSmThreads) small_kernel(SmallArgs a) {
    using S = typename std::conditional<MODE == MODE_FP64, double, float>::type;
    constexpr int TD = (TENSOR == T_OSEEN) ? T_OSEEN : T_RP;
    constexpr int I = small_block<MODE, R>();
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_end, s_cnt[2];   // s_end: the step in which a wait ran out somewhere in the cluster
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nt = a.nbl * I;                      // targets of this CTA
    const int WB = a.wb;                           // warps per target block
    const int lb = warp / WB, ws = warp % WB;      // (lb >= nbl: a warp without a block)
    double *s_v = reinterpret_cast<double *>(smem);
    double *s_sum = s_v + 3 * (nt + kSmMaxSplit);
    double *s_cor = s_sum + 3 * nt, *s_ahead = s_cor, *s_pd = s_cor, *s_x = s_cor;
    int *s_note = nullptr, *s_sort = nullptr;
    const int pd = a.jlen + nt;
    if constexpr (MODE != MODE_FP64) {
        s_ahead = s_cor + 3 * kSmNotes;
        s_pd = s_ahead + 3 * kSmAhead;
        s_note = reinterpret_cast<int *>(s_pd + 3 * pd);   // [2][kSmNotes]
        s_sort = s_note + 2 * kSmNotes;
        s_x = s_pd + 3 * pd + 3 * kSmNotes / 2;
    }
    S *s_src = reinterpret_cast<S *>(reinterpret_cast<double *>(smem) + small_words(MODE, a.jlen, nt, a.solo, a.n));
    S *s_tgt = s_src + 6 * a.jlen;
    S *s_red = s_tgt + 3 * nt;                     // [WB][6 or 3][nt]

    const int sp = static_cast<int>(blockIdx.x) % a.nsplit;   // = the CTA's rank in its cluster
    const int i0 = static_cast<int>(blockIdx.x) / a.nsplit * I, j0 = sp * a.jlen;
    const int jn = min(a.jlen, a.n - j0);          // (>= 1) sources of this split; the rest are padding
    const bool mine = i0 < a.row1 && i0 + nt > a.row0;   // some of the block's rows are wanted (uniform over a cluster)
    unsigned tag = 0;
    if (!a.solo && a.out == OUT_EULER && a.nsteps > 1) tag = *reinterpret_cast<volatile unsigned *>(a.sync);
    if (tid == 0) {
        s_end = 0x7fffffff;
        s_cnt[0] = s_cnt[1] = 0;
    }

    // forces of the sources, constant over the launch
    for (int q = tid; q < a.jlen; q += kSmThreads)
        for (int d = 0; d < 3; ++d) {
            S f = S(0);
            if (q < jn) {
                const size_t k = 3 * static_cast<size_t>(j0 + q) + d;
                f = static_cast<S>(a.f32 ? static_cast<double>(static_cast<const float *>(a.F)[k])
                                         : static_cast<const double *>(a.F)[k]);
            }
            s_src[(3 + d) * a.jlen + q] = f;
        }
    if (a.solo)
        for (int k = tid; k < 3 * a.n; k += kSmThreads) s_x[k] = a.x0[k];

    // phase B: one (row, component) of the rows sp rows .. of the block per thread; its
    // force and self term do not change during the launch
    const int er = tid / 3, ed = tid % 3, ei = i0 + sp * a.rows + er;
    const bool upd = er < a.rows && sp * a.rows + er < nt && ei < a.n;
    const size_t ek = 3 * static_cast<size_t>(ei) + ed;
    const bool row = ei >= a.row0 && ei < a.row1;   // (a row shard: the other rows keep their positions)
    double self = 0.0;   // F_i (mu_ii / mu0 = I); FP32C: minus the clamped self term the loop adds
    if (upd) {
        self = a.f32 ? static_cast<double>(static_cast<const float *>(a.F)[ek]) : static_cast<const double *>(a.F)[ek];
        if (a.out != OUT_EULER && row && !isfinite(self)) atomicOr(a.err, DEV_ERR_NONFINITE);
        if constexpr (MODE != MODE_FP64) {
            const float ri = rsqrt_sfu(a.pc.r2min_f), ri2 = __fmul_rn(ri, ri);
            const float A = TD == T_OSEEN ? __fmul_rn(a.pc.c1_f, ri)
                                          : __fmul_rn(ri, __fmaf_rn(a.pc.c3_f, ri2, a.pc.c1_f));
            self -= static_cast<double>(__fmul_rn(A, static_cast<float>(self)));
        }
    }
    // phase A's last part: the component sd of target st per thread, for the CTA that updates it
    const int sd = tid >> a.lnt, st = tid & (nt - 1), owner = st / a.rows;
    const uint32_t sdst =
        tid < 3 * nt && a.nsplit > 1
            ? cluster_addr(s_v + (static_cast<size_t>(sp) * 3 + sd) * a.rows + (st - owner * a.rows), owner)
            : 0u;
    double xe = upd && a.out == OUT_EULER ? a.x0[ek] : 0.0;
    const int passes = a.out == OUT_EULER ? a.nsteps : 1;

    for (int step = 0; step < passes; ++step) {
        double *x, *xn;
        if (a.stride) {
            x = a.x0 + step * a.stride;
            xn = x + a.stride;
        } else {
            x = (step & 1) ? a.x1 : a.x0;
            xn = (step & 1) ? a.x0 : a.x1;
        }
        if (a.solo || step == 0) __syncthreads();
        // ---- phase A: positions relative to particle 0, sources and targets
        const ulonglong2 *xb = a.xch + static_cast<size_t>(step & 1) * 3 * a.n;
        const int cur = step & 1;
        if (mine) {
            for (int q = tid; q < pd; q += kSmThreads) {
                const bool src = q < a.jlen;
                const int p = src ? j0 + q : i0 + q - a.jlen;
                S *dst = src ? s_src + q : s_tgt + (q - a.jlen);
                const int ld_dst = src ? a.jlen : nt;
                S v[3] = {static_cast<S>(src ? 1.0e18 : -1.0e18), S(0), S(0)};
                if (src ? q < jn : p < a.n) {
                    double org[3], u[3];
                    if (a.solo || step == 0) {
                        const double *from = a.solo ? s_x : x;
                        for (int d = 0; d < 3; ++d) {
                            org[d] = from[d];
                            u[d] = from[3 * static_cast<size_t>(p) + d];
                        }
                    } else if (!xch_get(a, xb, p, tag + step - 1, org, u) &&
                               *reinterpret_cast<volatile int *>(&s_end) >= step) {
                        // A wait ran out.  The cluster has to leave together, since its CTAs store
                        // into each other's shared memory (padding rows too, which no wait stands
                        // for): all are told this step before its barrier and leave at the check in
                        // the next one.  (Told earlier, its peers may be gone.  What the step
                        // computes from here is of no use, but in bounds.)
                        for (int r = 0; r < a.nsplit; ++r) cluster_store(cluster_addr(&s_end, r), step);
                    }
                    for (int d = 0; d < 3; ++d) {
                        u[d] -= org[d];
                        if constexpr (MODE != MODE_FP64) s_pd[d * pd + q] = u[d];
                        v[d] = static_cast<S>(PER ? wrap_coord(u[d], a.pc.Ld[d], a.pc.invLd[d]) : u[d]);
                    }
                }
                for (int d = 0; d < 3; ++d) dst[d * ld_dst] = v[d];
            }
        }
        __syncthreads();
        if (s_end < step) break;   // (the same for all threads of the cluster: a peer told now writes this step)
        const int nprev = step == 0 ? 0 : s_cnt[cur ^ 1];   // the last step's notes
        if (mine) {
            const SmallNear nr{reinterpret_cast<const float *>(s_src), reinterpret_cast<const float *>(s_tgt), s_pd,
                               a.jlen, nt, j0};
            if constexpr (MODE != MODE_FP64) {   // the last step's near pairs at the new positions
                if (warp == kSmWarps)
                    for (int m = lane; m < min(nprev, kSmAhead); m += 32) {
                        small_near<TENSOR, PER>(a, nr, s_note[(cur ^ 1) * kSmNotes + m], s_ahead + 3 * m);
                    }
            }
            if constexpr (MODE == MODE_FP64) {
                // lane = (target, source offset): iw targets, 32 / iw sources at a time
                if (lb < a.nbl) {
                    const int li = lane & (a.iw - 1), jo = lane / a.iw, js = 32 / a.iw;
                    const int t = lb * I + li, i = i0 + t;
                    const double xi = s_tgt[t], yi = s_tgt[nt + t], zi = s_tgt[2 * nt + t];
                    double ax = 0.0, ay = 0.0, az = 0.0;
                    for (int q = ws * js + jo; q < jn; q += WB * js)
                        small_pair64<TENSOR, PER>(xi, yi, zi, s_src[q], s_src[a.jlen + q], s_src[2 * a.jlen + q],
                                                  s_src[3 * a.jlen + q], s_src[4 * a.jlen + q],
                                                  s_src[5 * a.jlen + q], j0 + q == i, a, ax, ay, az);
                    for (int o = a.iw; o < a.span; o <<= 1) {
                        ax += __shfl_xor_sync(0xffffffffu, ax, o);
                        ay += __shfl_xor_sync(0xffffffffu, ay, o);
                        az += __shfl_xor_sync(0xffffffffu, az, o);
                    }
                    if (jo == 0) {
                        double *r = s_red + static_cast<size_t>(ws) * 3 * nt + t;
                        r[0] = ax;
                        r[nt] = ay;
                        r[2 * nt] = az;
                    }
                }
            } else {
                if (lb < a.nbl) {
                    f2 XI[R], YI[R], ZI[R], AX[R], AY[R], AZ[R];
#pragma unroll
                    for (int k = 0; k < R; ++k) {
                        const int t = lb * I + lane + 32 * k;
                        const float fx = s_tgt[t], fy = s_tgt[nt + t], fz = s_tgt[2 * nt + t];
                        XI[k] = pk2(fx, fx);
                        YI[k] = pk2(fy, fy);
                        ZI[k] = pk2(fz, fz);
                        AX[k] = AY[k] = AZ[k] = 0ull;
                    }
                    float hi[R][3] = {}, lo[R][3] = {};
                    auto fold = [&]() {
#pragma unroll
                        for (int k = 0; k < R; ++k) {
                            const f2 acc[3] = {AX[k], AY[k], AZ[k]};
                            for (int d = 0; d < 3; ++d) {
                                float u, v;
                                upk2(acc[d], u, v);
                                fold2(hi[k][d], lo[k][d], u);
                                fold2(hi[k][d], lo[k][d], v);
                            }
                            AX[k] = AY[k] = AZ[k] = 0ull;
                        }
                    };
                    int since = 0;
                    for (int q = 4 * ws; q < a.jlen; q += 4 * WB) {
                        f2 P[6][2];
#pragma unroll
                        for (int d = 0; d < 6; ++d) {
                            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(s_src + d * a.jlen + q);
                            P[d][0] = v.x;
                            P[d][1] = v.y;
                        }
                        float rr[R][4];
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int k = 0; k < R; ++k)
                                pair_f32x2_t<TD, true, true, PER>(XI[k], YI[k], ZI[k], P[0][h], P[1][h], P[2][h],
                                                                  P[3][h], P[4][h], P[5][h], a.c2, AX[k], AY[k],
                                                                  AZ[k], rr[k][2 * h], rr[k][2 * h + 1]);
                        float mn = 3.0e38f;
#pragma unroll
                        for (int k = 0; k < R; ++k)
                            mn = fminf(mn, fminf(fminf(rr[k][0], rr[k][1]), fminf(rr[k][2], rr[k][3])));
                        if (mn <= a.rscreen2) {   // rare: near pairs, and each target's self pair once
#pragma unroll
                            for (int k = 0; k < R; ++k)
#pragma unroll
                                for (int u = 0; u < 4; ++u) {
                                    const int t = lb * I + lane + 32 * k;
                                    if (rr[k][u] <= a.rscreen2 && q + u < jn && i0 + t < a.n && i0 + t != j0 + q + u) {
                                        const int m = atomicAdd(&s_cnt[cur], 1);
                                        if (m < kSmNotes) s_note[cur * kSmNotes + m] = (t << 16) | (q + u);
                                    }
                                }
                        }
                        if (++since == 16) {   // (at most 32 terms per packed lane between folds)
                            fold();
                            since = 0;
                        }
                    }
                    fold();
#pragma unroll
                    for (int k = 0; k < R; ++k)
                        for (int d = 0; d < 3; ++d) {
                            float *r = s_red + static_cast<size_t>(ws) * 6 * nt + lb * I + lane + 32 * k;
                            r[d * nt] = hi[k][d];
                            r[(3 + d) * nt] = lo[k][d];
                        }
                }
            }
            __syncthreads();
            int ne = 0;
            if constexpr (MODE != MODE_FP64) {
                ne = s_cnt[cur];
                const int *note = s_note + cur * kSmNotes, *prev = s_note + (cur ^ 1) * kSmNotes;
                if (ne <= kSmNotes) {
                    for (int m = kSmThreads - 1 - tid; m < ne; m += kSmThreads) {   // (the last warps first)
                        const int key = note[m];
                        int rank = 0, at = -1;
                        for (int k = 0; k < ne; ++k) rank += note[k] < key;
                        for (int k = 0; k < min(nprev, kSmAhead); ++k)
                            if (prev[k] == key) at = k;
                        rank = static_cast<int>(dbg_index(rank, kSmNotes, a.err));
                        s_sort[rank] = key >> 16;
                        if (at >= 0)
                            for (int d = 0; d < 3; ++d) s_cor[3 * rank + d] = s_ahead[3 * at + d];
                        else
                            small_near<TENSOR, PER>(a, nr, key, s_cor + 3 * rank);
                    }
                } else {
                    // The notes overflowed (a lattice whose indices follow its sites): four lanes
                    // of each target scan the CTA's sources again, 32 each at a time, and take
                    // the FP64 terms of those within reach together (a term at a time as they
                    // are met: 0.18 ms a step for 108 spheres of an fcc lattice); the lanes meet
                    // in a fixed tree.
                    for (int t4 = tid; t4 < 4 * nt; t4 += kSmThreads) {   // (whole warps)
                        const int t = t4 >> 2, sub = t4 & 3;
                        double sum[3] = {0.0, 0.0, 0.0};
                        for (int q0 = sub; q0 - sub < jn; q0 += 128) {
                            unsigned hit = 0;
                            for (int k = 0; k < 32; ++k) {
                                const int q = q0 + 4 * k;
                                if (q >= jn) break;
                                float dx = __fsub_rn(s_tgt[t], s_src[q]), dy = __fsub_rn(s_tgt[nt + t], s_src[a.jlen + q]),
                                      dz = __fsub_rn(s_tgt[2 * nt + t], s_src[2 * a.jlen + q]);
                                if (PER) {
                                    dx = min_image_f32(dx, a.pc.Lf[0], a.pc.invLf[0]);
                                    dy = min_image_f32(dy, a.pc.Lf[1], a.pc.invLf[1]);
                                    dz = min_image_f32(dz, a.pc.Lf[2], a.pc.invLf[2]);
                                }
                                if (__fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx))) <= a.rscreen2 &&
                                    j0 + q != i0 + t && i0 + t < a.n)
                                    hit |= 1u << k;
                            }
                            while (__any_sync(0xffffffffu, hit != 0)) {
                                if (hit) {
                                    double c[3];
                                    const int q = q0 + 4 * (__ffs(hit) - 1);
                                    hit &= hit - 1;
                                    if (small_near<TENSOR, PER>(a, nr, (t << 16) | q, c))
                                        for (int d = 0; d < 3; ++d) sum[d] += c[d];
                                }
                                __syncwarp();
                            }
                        }
                        for (int d = 0; d < 3; ++d) {
                            sum[d] += __shfl_xor_sync(0xffffffffu, sum[d], 1);
                            sum[d] += __shfl_xor_sync(0xffffffffu, sum[d], 2);
                            if (sub == 0) s_cor[3 * t + d] = sum[d];   // (nt <= kSmNotes)
                        }
                    }
                }
            }
            // the warps' sums: four lanes take the warps w = 0, 1, 2, 3 mod 4 of an output each
            // and meet in a fixed tree
            for (int o4 = tid; o4 < 12 * nt; o4 += kSmThreads) {   // (12 nt: a multiple of 32)
                const int o = o4 >> 2, sub = o4 & 3, d = o >> a.lnt, t = o & (nt - 1);
                if constexpr (MODE == MODE_FP64) {
                    double v = 0.0;
                    for (int w = sub; w < WB; w += 4) v += s_red[(static_cast<size_t>(w) * 3 + d) * nt + t];
                    if (WB > 1) v += __shfl_xor_sync(0xffffffffu, v, 1);
                    if (WB > 2) v += __shfl_xor_sync(0xffffffffu, v, 2);
                    if (sub == 0) s_sum[o] = v;
                } else {
                    float h = 0.0f, l = 0.0f;
                    for (int w = sub; w < WB; w += 4) {
                        const float *r = s_red + static_cast<size_t>(w) * 6 * nt + t;
                        fold2(h, l, r[d * nt]);
                        l = __fadd_rn(l, r[(3 + d) * nt]);
                    }
#pragma unroll
                    for (int m = 1; m <= 2; m <<= 1) {
                        const float h2 = __shfl_xor_sync(0xffffffffu, h, m), l2 = __shfl_xor_sync(0xffffffffu, l, m);
                        fold2(h, l, h2);
                        l = __fadd_rn(l, l2);
                    }
                    if (sub == 0) reinterpret_cast<float2 *>(s_sum)[o] = make_float2(h, l);
                }
            }
            __syncthreads();
            // the near corrections in (target, source) order join; FP32C sums travel as (hi, lo)
            if (tid < 3 * nt) {   // (3 nt <= 384)
                double v = s_sum[tid];
                if constexpr (MODE != MODE_FP64) {
                    if (ne) {
                        double c = 0.0;
                        bool any = ne > kSmNotes;
                        if (any) c = s_cor[3 * st + sd];
                        else
                            for (int k = 0; k < ne; ++k)
                                if (s_sort[k] == st) {
                                    c += s_cor[3 * k + sd];
                                    any = true;
                                }
                        if (any) {
                            float2 q = reinterpret_cast<float2 *>(s_sum)[tid];
                            const float ch = static_cast<float>(c);
                            fold2(q.x, q.y, ch);
                            q.y = __fadd_rn(q.y, static_cast<float>(c - static_cast<double>(ch)));
                            reinterpret_cast<float2 *>(s_sum)[tid] = q;
                            v = s_sum[tid];
                        }
                    }
                }
                if (a.nsplit > 1) cluster_store(sdst, v);
                else s_v[sd * a.rows + st] = v;
            }
            if (tid == 0) s_cnt[cur ^ 1] = 0;   // (read above; the next step's notes)
        }
        if (a.nsplit > 1) cluster_barrier();
        else __syncthreads();
        // ---- phase B
        if (upd && !row) {
            if (a.out == OUT_EULER) xn[ek] = x[ek];   // (row shards: single steps only)
        } else if (upd) {
            double v = self;
            if constexpr (MODE == MODE_FP64) {
                double sum = s_v[ed * a.rows + er];
                for (int s = 1; s < a.nsplit; ++s) sum += s_v[(s * 3 + ed) * a.rows + er];
                v = __fma_rn(a.pc.c1_d, sum, v);
            } else {
                const float2 *q = reinterpret_cast<const float2 *>(s_v) + ed * a.rows + er;
                float h = q[0].x, l = q[0].y;
                for (int s = 1; s < a.nsplit; ++s) {
                    const float2 w = q[3 * s * a.rows];
                    fold2(h, l, w.x);
                    l = __fadd_rn(l, w.y);
                }
                v += static_cast<double>(h) + static_cast<double>(l);
            }
            if (a.out == OUT_F32) {
                static_cast<float *>(a.vout)[ek - 3 * static_cast<size_t>(a.row0)] = static_cast<float>(a.pc.mu0 * v);
            } else if (a.out == OUT_F64) {
                static_cast<double *>(a.vout)[ek - 3 * static_cast<size_t>(a.row0)] = a.pc.mu0 * v;
            } else {
                xe += a.dt * (a.pc.mu0 * v);   // this thread's FP64 coordinate, kept from step to step
                if (!isfinite(xe)) atomicOr(a.err, DEV_ERR_NONFINITE);
                if (a.solo) s_x[ek] = xe;
                else if (step + 1 < passes) xch_put(a.xch + static_cast<size_t>(cur ^ 1) * 3 * a.n + ek, xe, tag + step);
                if (a.stride || step + 1 == passes) xn[ek] = xe;
            }
        }
    }
    // (no CTA stores into another's shared memory after the last step's cluster barrier, which all
    // CTAs of the cluster have passed)
    if (!a.solo && passes > 1 && tid == 0) {   // the last CTA out: the next launch's tags are new ones
        __threadfence();
        if (atomicAdd(a.sync + 2, 1u) == gridDim.x - 1) {
            a.sync[0] = tag + static_cast<unsigned>(passes);
            a.sync[1] = 0u;
            a.sync[2] = 0u;
        }
    }
}

template <int MODE, int R>
static const void *small_fn_r(int tensor, bool per) {
    switch (tensor) {
        case T_RPY: return per ? reinterpret_cast<const void *>(&small_kernel<T_RPY, MODE, true, R>)
                               : reinterpret_cast<const void *>(&small_kernel<T_RPY, MODE, false, R>);
        case T_RP: return per ? reinterpret_cast<const void *>(&small_kernel<T_RP, MODE, true, R>)
                              : reinterpret_cast<const void *>(&small_kernel<T_RP, MODE, false, R>);
        default: return per ? reinterpret_cast<const void *>(&small_kernel<T_OSEEN, MODE, true, R>)
                            : reinterpret_cast<const void *>(&small_kernel<T_OSEEN, MODE, false, R>);
    }
}
static const void *small_fn(const sd_handle *h) {
    const bool per = h->pc.periodic != 0;
    if (h->mode == MODE_FP64) return small_fn_r<MODE_FP64, 1>(h->tensor, per);
    return h->small.R == 1 ? small_fn_r<MODE_FP32C, 1>(h->tensor, per) : small_fn_r<MODE_FP32C, 2>(h->tensor, per);
}

// Launch configuration: clusters of `split` CTAs, cooperative when the grid meets.
static void small_config(const sd_handle *h, cudaLaunchConfig_t &cfg, cudaLaunchAttribute (&at)[2], cudaStream_t st,
                         bool coop) {
    const SmallGeom &g = h->small;
    cfg.gridDim = dim3(g.grid);
    cfg.blockDim = dim3(kSmThreads);
    cfg.dynamicSmemBytes = g.smem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = g.split;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeCooperative;
    at[1].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = coop ? 2 : 1;
}

// Which systems take this path: the all-pairs kernel left to the library (a caller that
// names one gets it) and resolved to the directed one (dense_setup; on 152 SMs FP32C n <= 3,072,
// FP64 n <= 1,408: from there on using every pair once pays for the further kernels), and
// forces that do not change with the positions.
cudaError_t small_setup(sd_handle *h) {
    SmallGeom &g = h->small;
    g = SmallGeom{};
    if (h->cfg.dense_kernel != SD_DENSE_AUTO || h->geom.sym || !h->forces_const || h->mode == MODE_FP32 || h->n < 1)
        return cudaSuccess;
    int coop = 0;
    cudaError_t e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, h->device);
    if (e != cudaSuccess || !coop) return e;
    const bool f64 = h->mode == MODE_FP64;
    const int n = h->n;
    g.solo = n <= (f64 ? kSmSoloFP64 : kSmSoloFP32);
    // (FP32C near pairs cost one SM some 900 cycles a warp of them: a dense box takes more SMs)
    if (!f64 && h->pc.Ld[0] > 0.0 && h->pc.Ld[1] > 0.0 && h->pc.Ld[2] > 0.0) {
        const double rn = h->r_near;
        const double close = 4.18879 * rn * rn * rn * n / (h->pc.Ld[0] * h->pc.Ld[1] * h->pc.Ld[2]);
        if (n * close > kSmNotes) g.solo = 0;
        if (n * close > kSmDense) return cudaSuccess;
    }
    if (f64)
        while (g.iw > 1 && g.iw / 2 >= n) g.iw /= 2;
    bool tried[3][kSmMaxSplit + 1] = {};
    for (;;) {
        // targets per thread and j-splits: the least work per SM, of those whose clusters
        // all fit at once
        long long best = -1;
        g.R = g.split = 1;
        for (int R = 1; R <= (f64 || g.solo ? 1 : 2); ++R) {
            const int nib = (n + 32 * R - 1) / (32 * R);
            for (int s = 1; s <= (g.solo ? 1 : kSmMaxSplit) && (g.solo || nib * s <= h->num_sms); ++s) {
                if (tried[R][s]) continue;
                const int jlen = ((n + s - 1) / s + 3) & ~3;
                const long long quads = (jlen / 4 + kSmWarps - 1) / kSmWarps;
                // (per step: packed pair terms, a round of 300 cycles each, and the positions
                // fetched, one round of 500 threads about 600 cycles)
                const long long cost = f64 ? static_cast<long long>(jlen) * 1000 + s
                                           : quads * R * 300000 + (jlen + 32 * R) * 1200LL + s;
                if (best < 0 || cost < best) {
                    best = cost;
                    g.R = R;
                    g.split = s;
                }
            }
        }
        if (best < 0) return cudaSuccess;
        tried[g.R][g.split] = true;
        g.nib = (n + 32 * g.R - 1) / (32 * g.R);
        g.nbl = g.solo ? (g.nib == 3 ? 4 : g.nib) : 1;   // (a power of two)
        g.jlen = ((n + g.split - 1) / g.split + 3) & ~3;
        if ((n + g.jlen - 1) / g.jlen != g.split) continue;   // (no empty split)
        // no more warps per block than it has groups of sources (four sources; FP64 32 / iw)
        const int groups = f64 ? (g.jlen + 32 / g.iw - 1) / (32 / g.iw) : g.jlen / 4;
        g.wb = std::max(1, std::min(kSmWarps / g.nbl, groups));
        g.grid = g.solo ? 1 : g.nib * g.split;
        g.rows = (g.nbl * 32 * g.R + g.split - 1) / g.split;
        g.smem = small_smem(h->mode, g.R, g.jlen, g.nbl, g.wb, g.solo, n);
        const void *fn = small_fn(h);
        size_t limit = 0;
        e = allow_smem(fn, limit);
        if (e != cudaSuccess) return e;
        if (g.smem > limit) continue;
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at[2];
        small_config(h, cfg, at, nullptr, false);
        int clusters = 0;
        e = cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg);
        if (e != cudaSuccess) return e;
        g.on = clusters * g.split >= g.grid;
        if (g.on) return cudaSuccess;
    }
}

// out = OUT_F32 / OUT_F64: vout = rows [row0, row1) of mu(x0) F.  OUT_EULER: nsteps steps
// (at most kSmMaxSteps a launch) from x0, alternating with x1, or (stride > 0) from row
// to row of x0.
cudaError_t launch_small(sd_handle *h, cudaStream_t st, int out, double *x0, double *x1, size_t stride, const void *F,
                         int f32, void *vout, double dt, int64_t nsteps, int row0, int row1) {
    const SmallGeom &g = h->small;
    SmallArgs a{};
    a.F = F;
    a.f32 = f32;
    a.vout = vout;
    a.out = out;
    a.n = h->n;
    a.rows = g.rows;
    a.lnt = 5;
    while ((1 << a.lnt) < g.nbl * 32 * g.R) ++a.lnt;
    a.nsplit = g.split;
    a.jlen = g.jlen;
    a.nbl = g.nbl;
    a.wb = g.wb;
    a.iw = a.span = g.iw;
    while (a.span < 32 && a.span < g.iw * g.jlen) a.span *= 2;
    a.solo = g.solo;
    a.row0 = row0;
    a.row1 = row1;
    a.dt = dt;
    a.rnear2 = h->r_near * h->r_near;
    a.rscreen2 = static_cast<float>(1.0201 * h->r_near * h->r_near);
    a.pc = h->pc;
    a.c2 = pair_const2(h->pc, h->n);
    a.sync = h->small_sync;
    a.xch = h->small_xch;
    a.err = h->d_err;
    a.wd = h->watchdog;
    a.stride = stride;
    const void *fn = small_fn(h);
    int64_t left = out == OUT_EULER ? nsteps : 1;
    while (left > 0) {
        const int k = static_cast<int>(std::min<int64_t>(left, h->prof.on ? 1 : kSmMaxSteps));
        a.x0 = x0;
        a.x1 = x1;
        a.nsteps = k;
        void *args[] = {&a};
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at[2];
        small_config(h, cfg, at, st, !g.solo && out == OUT_EULER && k > 1);
        prof_begin(h, SD_KERNEL_DENSE, st);
        const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
        prof_end(h, SD_KERNEL_DENSE, st);
        if (e != cudaSuccess) return e;
        ++h->launches;
        if (stride) x0 += static_cast<size_t>(k) * stride;
        else if (k & 1) std::swap(x0, x1);
        left -= k;
    }
    return cudaSuccess;
}

}  // namespace sd
