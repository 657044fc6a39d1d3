// vjp.cu -- vector-Jacobian products of v(x, F) = mu(x) F (derivative of
// Sec. 2.2, Eq. rotneMobility; the paper has no adjoint):
//
//   (mu W)_i  = mu0 [ W_i + sum_{j != i} (A W_j + B (r.W_j) r) ]
//   gX_i      = mu0 sum_{j != i} grad_r [ W_i.T^(r) F_j + W_j.T^(r) F_i ],  r = x_i - x_j
//
// with T^ = T/mu0 = A I + B r r^T (pair.cuh).  mu is symmetric, so mu^T W = mu W
// is the force gradient.  One all-pairs kernel evaluates both sums from the same
// r, 1/r and tensor profile, each unordered pair once (mu_ij = mu_ji, and the pair's
// gradient with respect to x_j is minus that with respect to x_i); the layout is
// dense_sym_kernel's (block pairs over a persistent grid, bulk-copied source blocks of
// positions, forces and cotangents, source sums handed on by shuffle, per-tile TwoSum
// folds, fixed-order slots).  Beside it, the pairs closer than r_near, taken from the
// near pass's or the Verlet steps' candidate list, get exact FP64 values minus what the
// all-pairs kernel adds for them; the epilogue sums and swaps the self term.
#include <algorithm>
#include "neighbours.cuh"

namespace sd {

template <int MODE>
struct VjpT {
    using V4 = float4;
};
template <>
struct VjpT<MODE_FP64> {
    using V4 = dbl4;
};

// Above kVjpSymN particles, where the source-side sums of every block pair would take GBs,
// the directed kernels: FP64 (plain FP64 sums, divided by c1) and vjp2_kernel below.
template <int TENSOR, bool PER>
__global__ void __launch_bounds__(kNT) vjp_kernel(const dbl4 *__restrict__ pos, const dbl4 *__restrict__ frc,
                                                  const dbl4 *__restrict__ wv,
                                                  double *__restrict__ partM, double *__restrict__ partG, int npad,
                                                  DenseGeom g, PairConst c, int *__restrict__ err, long long wd) {
    using V4 = dbl4;
    constexpr int R = kRV;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ int s_abort;
    V4 *s_pos = reinterpret_cast<V4 *>(smem);
    V4 *s_frc = s_pos + 2 * g.J;
    V4 *s_w = s_frc + 2 * g.J;

    const int tid = threadIdx.x;
    const long long T = static_cast<long long>(g.nIB) * g.nJT;
    const long long t0 = static_cast<long long>(blockIdx.x) * g.chunk;
    const long long t1 = (t0 + g.chunk < T) ? t0 + g.chunk : T;
    if (t0 >= t1) return;
    const uint32_t tile_bytes = static_cast<uint32_t>(g.J * sizeof(V4));

    int issued0 = 0, issued1 = 0, waited0 = 0, waited1 = 0;
    if (tid == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        s_abort = 0;
        fence_barrier_init();
    }
    __syncthreads();
    auto issue = [&](long long t, int stg) {
        const size_t jt = static_cast<size_t>(t % g.nJT);
        mbar_arrive_expect_tx(&bars[stg], 3 * tile_bytes);
        bulk_g2s(s_pos + stg * g.J, pos + jt * g.J, tile_bytes, &bars[stg]);
        bulk_g2s(s_frc + stg * g.J, frc + jt * g.J, tile_bytes, &bars[stg]);
        bulk_g2s(s_w + stg * g.J, wv + jt * g.J, tile_bytes, &bars[stg]);
        if (stg == 0) ++issued0; else ++issued1;
    };
    if (tid == 0)
        for (int q = 0; q < 2 && t0 + q < t1; ++q) issue(t0 + q, q);

    double X[R][9], m[R][3], gg[R][3];
    int cur_ib = -1;
    bool aborted = false;

    auto flush = [&](int ib) {
        const int slot = static_cast<int>(blockIdx.x) - geom_first(g, ib);
        double *dM = partM + static_cast<size_t>(slot) * 3 * npad;
        double *dG = partG + static_cast<size_t>(slot) * 3 * npad;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const size_t i = static_cast<size_t>(ib) * g.I + tid + k * kNT;
            for (int d = 0; d < 3; ++d) {
                dM[d * static_cast<size_t>(npad) + i] = m[k][d];
                dG[d * static_cast<size_t>(npad) + i] = gg[k][d];
            }
        }
    };

    for (long long t = t0; t < t1; ++t) {
        const int ib = static_cast<int>(t / g.nJT);
        if (ib != cur_ib) {
            if (cur_ib >= 0) flush(cur_ib);
            cur_ib = ib;
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const size_t i = static_cast<size_t>(ib) * g.I + tid + k * kNT;
                const V4 p = pos[i], f = frc[i], w = wv[i];
                const double v[9] = {p.x, p.y, p.z, f.x, f.y, f.z, w.x, w.y, w.z};
                for (int d = 0; d < 9; ++d) X[k][d] = v[d];
                for (int d = 0; d < 3; ++d) m[k][d] = gg[k][d] = 0.0;
            }
        }
        const int q = static_cast<int>(t - t0);
        const int st = q & 1;
        if (!aborted) {
            if (mbar_wait_bounded(&bars[st], (q >> 1) & 1, wd)) {
                if (tid == 0) { if (st == 0) ++waited0; else ++waited1; }
            } else {
                atomicOr(err, DEV_ERR_TIMEOUT);
                s_abort = 1;
            }
        }
        const V4 *P = s_pos + st * g.J;
        const V4 *Fq = s_frc + st * g.J;
        const V4 *Wq = s_w + st * g.J;
        for (int jj = 0; jj < g.J; ++jj) {
            const V4 p = P[jj], f = Fq[jj], w = Wq[jj];
            const double v[9] = {p.x, p.y, p.z, f.x, f.y, f.z, w.x, w.y, w.z};
#pragma unroll
            for (int k = 0; k < R; ++k) vjp_sym_f64<TENSOR, PER, false>(X[k], v, c, m[k], gg[k], m[k], gg[k]);
        }
        __syncthreads();
        aborted = s_abort != 0;
        if (tid == 0 && !aborted && t + 2 < t1) issue(t + 2, st);
    }
    flush(cur_ib);
    if (tid == 0) {
        for (int k = waited0; k < issued0; ++k)
            if (!mbar_wait_bounded(&bars[0], k & 1, drain_limit(wd))) atomicOr(err, DEV_ERR_TIMEOUT);
        for (int k = waited1; k < issued1; ++k)
            if (!mbar_wait_bounded(&bars[1], k & 1, drain_limit(wd))) atomicOr(err, DEV_ERR_TIMEOUT);
    }
}

// FP32C: the same sums with the pair terms packed over pairs of sources.  The j-tiles
// are staged as nine float arrays (x, y, z, Fx, Fy, Fz, Wx, Wy, Wz: nine bulk copies),
// so two consecutive j's form one 64-bit operand and every instruction of
// vjp_pair_f32x2 evaluates (i, j) and (i, j + 1): half the issued instructions of the
// scalar loop (N = 4,096: 45 us against 48).  Each thread owns R targets, duplicated
// into both lanes; its packed
// accumulators sum even and odd j's separately, and both lanes are folded into (hi, lo)
// TwoSum accumulators in shared memory after every tile.  Slots are (hi, lo) float
// pairs, as the FP32C epilogue reads them.
// Targets per thread of the packed FP32C VJP kernel.  One keeps it at about 120
// registers (4 CTAs per SM); two took 140 and were slower at N = 4,096 (50 against 45 us).
#ifndef SD_VJP2_R
#define SD_VJP2_R 1
#endif
constexpr int kRV2 = SD_VJP2_R;

template <int TENSOR, bool PER>
__global__ void __launch_bounds__(kNT) vjp2_kernel(const float *__restrict__ pos, const float *__restrict__ frc,
                                                   const float *__restrict__ wv, double *__restrict__ partM,
                                                   double *__restrict__ partG, int npad, DenseGeom g, VjpConst2 c,
                                                   int *__restrict__ err, long long wd) {
    constexpr int R = kRV2;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ int s_abort;
    float *s_tile = reinterpret_cast<float *>(smem);   // [2 stages][9 arrays][J]
    float *s_acc = s_tile + 18 * g.J;                   // [R][12][kNT]: M hi(3) lo(3), G hi(3) lo(3)

    const int tid = threadIdx.x;
    const long long T = static_cast<long long>(g.nIB) * g.nJT;
    const long long t0 = static_cast<long long>(blockIdx.x) * g.chunk;
    const long long t1 = (t0 + g.chunk < T) ? t0 + g.chunk : T;
    if (t0 >= t1) return;
    const uint32_t arr_bytes = static_cast<uint32_t>(g.J * sizeof(float));

    int issued0 = 0, issued1 = 0, waited0 = 0, waited1 = 0;   // bookkeeping of thread 0 only
    if (tid == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        s_abort = 0;
        fence_barrier_init();
    }
    __syncthreads();
    auto issue = [&](long long t, int stg) {
        const size_t j0 = static_cast<size_t>(t % g.nJT) * g.J;
        float *dst = s_tile + stg * 9 * g.J;
        mbar_arrive_expect_tx(&bars[stg], 9 * arr_bytes);
        for (int a = 0; a < 3; ++a) {
            bulk_g2s(dst + a * g.J, pos + a * static_cast<size_t>(npad) + j0, arr_bytes, &bars[stg]);
            bulk_g2s(dst + (3 + a) * g.J, frc + a * static_cast<size_t>(npad) + j0, arr_bytes, &bars[stg]);
            bulk_g2s(dst + (6 + a) * g.J, wv + a * static_cast<size_t>(npad) + j0, arr_bytes, &bars[stg]);
        }
        if (stg == 0) ++issued0; else ++issued1;
    };
    if (tid == 0)
        for (int q = 0; q < 2 && t0 + q < t1; ++q) issue(t0 + q, q);

    f2 XI[R], YI[R], ZI[R], FI[R][3], WI[R][3];
    int cur_ib = -1;
    bool aborted = false;

    auto flush = [&](int ib) {
        const int slot = static_cast<int>(blockIdx.x) - geom_first(g, ib);
        float2 *dM = reinterpret_cast<float2 *>(partM) + static_cast<size_t>(slot) * 3 * npad;
        float2 *dG = reinterpret_cast<float2 *>(partG) + static_cast<size_t>(slot) * 3 * npad;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const size_t i = static_cast<size_t>(ib) * g.I + tid + k * kNT;
            const float *q = s_acc + k * 12 * kNT + tid;
            for (int d = 0; d < 3; ++d) {
                dM[d * static_cast<size_t>(npad) + i] = make_float2(q[d * kNT], q[(3 + d) * kNT]);
                dG[d * static_cast<size_t>(npad) + i] = make_float2(q[(6 + d) * kNT], q[(9 + d) * kNT]);
            }
        }
    };

    for (long long t = t0; t < t1; ++t) {
        const int ib = static_cast<int>(t / g.nJT);
        if (ib != cur_ib) {
            if (cur_ib >= 0) flush(cur_ib);
            cur_ib = ib;
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const size_t i = static_cast<size_t>(ib) * g.I + tid + k * kNT;
                const float x = pos[i], y = pos[npad + i], z = pos[2 * static_cast<size_t>(npad) + i];
                XI[k] = pk2(x, x);
                YI[k] = pk2(y, y);
                ZI[k] = pk2(z, z);
                for (int d = 0; d < 3; ++d) {
                    const float fv = frc[d * static_cast<size_t>(npad) + i], wvv = wv[d * static_cast<size_t>(npad) + i];
                    FI[k][d] = pk2(fv, fv);
                    WI[k][d] = pk2(wvv, wvv);
                }
                for (int e = 0; e < 12; ++e) s_acc[(k * 12 + e) * kNT + tid] = 0.0f;
            }
        }
        const int q = static_cast<int>(t - t0);
        const int st = q & 1;
        if (!aborted) {
            if (mbar_wait_bounded(&bars[st], (q >> 1) & 1, wd)) {
                if (tid == 0) { if (st == 0) ++waited0; else ++waited1; }
            } else {
                atomicOr(err, DEV_ERR_TIMEOUT);
                s_abort = 1;
            }
        }
        const float *src = s_tile + st * 9 * g.J;
        f2 M[R][3], G[R][3];
#pragma unroll
        for (int k = 0; k < R; ++k)
            for (int d = 0; d < 3; ++d) M[k][d] = G[k][d] = 0ull;
#pragma unroll 2
        for (int jj = 0; jj < g.J; jj += 4) {
            f2 P[9][2];   // four sources: two packed pairs per array
#pragma unroll
            for (int a = 0; a < 9; ++a) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(src + a * g.J + jj);
                P[a][0] = v.x;
                P[a][1] = v.y;
            }
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2)
#pragma unroll
                for (int k = 0; k < R; ++k)
                    vjp_pair_f32x2<TENSOR, PER>(XI[k], YI[k], ZI[k], FI[k][0], FI[k][1], FI[k][2], WI[k][0], WI[k][1],
                                                WI[k][2], P[0][h2], P[1][h2], P[2][h2], P[3][h2], P[4][h2], P[5][h2],
                                                P[6][h2], P[7][h2], P[8][h2], c, M[k], G[k]);
        }
#pragma unroll
        for (int k = 0; k < R; ++k)
            for (int d = 0; d < 3; ++d) {
                float lo, hi;
                float *q0 = s_acc + (k * 12 + d) * kNT + tid;   // M hi; M lo at +3 kNT
                upk2(M[k][d], lo, hi);
                float h = q0[0], l = q0[3 * kNT];
                fold2(h, l, lo);
                fold2(h, l, hi);
                q0[0] = h;
                q0[3 * kNT] = l;
                float *q1 = s_acc + (k * 12 + 6 + d) * kNT + tid;   // G hi; G lo at +3 kNT
                upk2(G[k][d], lo, hi);
                h = q1[0];
                l = q1[3 * kNT];
                fold2(h, l, lo);
                fold2(h, l, hi);
                q1[0] = h;
                q1[3 * kNT] = l;
            }
        __syncthreads();   // every thread is done with stage st
        aborted = s_abort != 0;
        if (tid == 0 && !aborted && t + 2 < t1) issue(t + 2, st);
    }
    flush(cur_ib);
    if (tid == 0) {
        for (int k = waited0; k < issued0; ++k)
            if (!mbar_wait_bounded(&bars[0], k & 1, drain_limit(wd))) atomicOr(err, DEV_ERR_TIMEOUT);
        for (int k = waited1; k < issued1; ++k)
            if (!mbar_wait_bounded(&bars[1], k & 1, drain_limit(wd))) atomicOr(err, DEV_ERR_TIMEOUT);
    }
}

// ---------------------------------------------------------------- symmetric kernels

// (ib, jb) of tile t of the upper triangle.
__device__ __forceinline__ void sym_tile_at(const DenseGeom &g, long long t, int &ib, int &jb) {
    const int nb = g.nIB;
    const double q = 2.0 * nb + 1.0;
    ib = static_cast<int>(0.5 * (q - sqrt(q * q - 8.0 * static_cast<double>(t))));
    ib = ib < 0 ? 0 : (ib > nb - 1 ? nb - 1 : ib);
    while (ib > 0 && geom_rowstart(g, ib) > t) --ib;
    while (ib + 1 < nb && geom_rowstart(g, ib + 1) <= t) ++ib;
    jb = ib + static_cast<int>(t - geom_rowstart(g, ib));
}

// FP32C.  Bound by the FP32 pipe (76 packed operations for two unordered pairs; the directed
// vjp2_kernel takes 128).  Blocks of B particles, R = 2 targets per lane (with one, the
// twelve words of source sums that a step hands on by shuffle weigh twice as much; more do
// not fit the registers), walked as in dense_sym_kernel; diagonal tiles run the directed
// pair.  Target sums are folded into (hi, lo) sums after every 64 sources; a tile's source sums
// are added over the warps in fixed order and go to its own rows of jpart in FP32.
// N = 4,096: 42 us directed, 31 (55% of the pipe: 3.5 CTAs of two warps an SM); whole call at
// 4,096 / 16,384: 96 / 716 -> 57 / 393 us (with one target per lane and four warps 59 at 4,096).
template <int TENSOR, bool PER, int B, int NT>
__global__ void __launch_bounds__(NT) vjp_sym_kernel(const float *__restrict__ pos, const float *__restrict__ frc,
                                                     const float *__restrict__ wv, double *__restrict__ partM,
                                                     double *__restrict__ partG, float *__restrict__ jpart, int npad,
                                                     DenseGeom g, VjpConst2 c, int *__restrict__ err, long long wd) {
    constexpr int R = B / NT, NW = NT / 32, S = B / 2;   // S: packets per array
    static_assert(B == NT * R && B % 64 == 0, "whole packets of 64 sources");
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ int s_abort;
    float *s_tile = reinterpret_cast<float *>(smem);   // [2 stages][9 arrays][B]
    float *s_acc = s_tile + 18 * B;                     // [R][12][NT]: M hi(3) lo(3), G hi(3) lo(3)
    float *s_jacc = s_acc + R * 12 * NT;                // [NW][6][B]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long t0 = static_cast<long long>(blockIdx.x) * g.chunk;
    const long long t1 = (t0 + g.chunk < g.nT) ? t0 + g.chunk : g.nT;
    if (t0 >= t1) return;
    constexpr uint32_t arr_bytes = B * sizeof(float);
    int ib, jb;
    sym_tile_at(g, t0, ib, jb);
    int issued0 = 0, issued1 = 0, waited0 = 0, waited1 = 0;   // bookkeeping of thread 0 only
    if (tid == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        s_abort = 0;
        fence_barrier_init();
    }
    __syncthreads();
    int qi = ib, qj = jb;   // next tile to stage (thread 0)
    auto issue = [&](int stg) {
        const size_t j0 = static_cast<size_t>(qj) * B;
        float *dst = s_tile + stg * 9 * B;
        mbar_arrive_expect_tx(&bars[stg], 9 * arr_bytes);
        for (int a = 0; a < 3; ++a) {
            const size_t off = a * static_cast<size_t>(npad) + j0;
            bulk_g2s(dst + a * B, pos + off, arr_bytes, &bars[stg]);
            bulk_g2s(dst + (3 + a) * B, frc + off, arr_bytes, &bars[stg]);
            bulk_g2s(dst + (6 + a) * B, wv + off, arr_bytes, &bars[stg]);
        }
        if (stg == 0) ++issued0; else ++issued1;
        if (++qj == g.nIB) { ++qi; qj = qi; }
    };
    if (tid == 0)
        for (int q = 0; q < 2 && t0 + q < t1; ++q) issue(q);

    f2 XI[R], YI[R], ZI[R], FI[R][3], WI[R][3], M[R][3], G[R][3];
    int cur_ib = -1;
    bool aborted = false;
    auto flush = [&](int row) {
        const size_t slot = blockIdx.x - geom_first(g, row);
        float2 *dM = reinterpret_cast<float2 *>(partM) + slot * 3 * npad;
        float2 *dG = reinterpret_cast<float2 *>(partG) + slot * 3 * npad;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const size_t i = static_cast<size_t>(row) * B + tid + k * NT;
            const float *q = s_acc + k * 12 * NT + tid;
            for (int d = 0; d < 3; ++d) {
                dM[d * static_cast<size_t>(npad) + i] = make_float2(q[d * NT], q[(3 + d) * NT]);
                dG[d * static_cast<size_t>(npad) + i] = make_float2(q[(6 + d) * NT], q[(9 + d) * NT]);
            }
        }
    };
    for (long long t = t0; t < t1; ++t) {
        if (ib != cur_ib) {
            if (cur_ib >= 0) flush(cur_ib);
            cur_ib = ib;
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const size_t i = static_cast<size_t>(ib) * B + tid + k * NT, N = npad;
                XI[k] = pk2(pos[i], pos[i]);
                YI[k] = pk2(pos[N + i], pos[N + i]);
                ZI[k] = pk2(pos[2 * N + i], pos[2 * N + i]);
                for (int d = 0; d < 3; ++d) {
                    const float fv = frc[d * N + i], w = wv[d * N + i];
                    FI[k][d] = pk2(fv, fv);
                    WI[k][d] = pk2(w, w);
                }
                for (int e = 0; e < 12; ++e) s_acc[(k * 12 + e) * NT + tid] = 0.0f;
            }
        }
        const int q = static_cast<int>(t - t0), st = q & 1;
        if (!aborted) {
            if (mbar_wait_bounded(&bars[st], (q >> 1) & 1, wd)) {
                if (tid == 0) { if (st == 0) ++waited0; else ++waited1; }
            } else {
                atomicOr(err, DEV_ERR_TIMEOUT);
                s_abort = 1;
            }
        }
#pragma unroll
        for (int k = 0; k < R; ++k)
            for (int d = 0; d < 3; ++d) M[k][d] = G[k][d] = 0ull;
        auto fold = [&]() {   // both lanes of the packed sums into the (hi, lo) sums
#pragma unroll
            for (int k = 0; k < R; ++k)
                for (int d = 0; d < 6; ++d) {
                    float lo, hi;
                    float *qa = s_acc + (k * 12 + (d < 3 ? d : 3 + d)) * NT + tid;   // hi; lo at + 3 NT
                    f2 &p = d < 3 ? M[k][d] : G[k][d - 3];
                    upk2(p, lo, hi);
                    p = 0ull;
                    float h = qa[0], l = qa[3 * NT];
                    fold2(h, l, lo);
                    fold2(h, l, hi);
                    qa[0] = h;
                    qa[3 * NT] = l;
                }
        };
        const bool diag = ib == jb;
        const f2 *sp = reinterpret_cast<const f2 *>(s_tile + st * 9 * B);
        if (diag) {
#pragma unroll 1
            for (int p = 0; p < S; ++p) {
                if (p && (p & 31) == 0) fold();
                f2 P[9];
#pragma unroll
                for (int a = 0; a < 9; ++a) P[a] = sp[a * S + p];
#pragma unroll
                for (int k = 0; k < R; ++k)
                    vjp_pair_f32x2<TENSOR, PER>(XI[k], YI[k], ZI[k], FI[k][0], FI[k][1], FI[k][2], WI[k][0], WI[k][1],
                                                WI[k][2], P[0], P[1], P[2], P[3], P[4], P[5], P[6], P[7], P[8], c,
                                                M[k], G[k]);
            }
        } else {
            const int nxt = (lane + 1) & 31;
            f2 *jw = reinterpret_cast<f2 *>(s_jacc + warp * 6 * B);
#pragma unroll 1
            for (int gq = 0; gq < B / 64; ++gq) {
                f2 JM[3] = {0ull, 0ull, 0ull}, JG[3] = {0ull, 0ull, 0ull};
#pragma unroll 2
                for (int m = 0; m < 32; ++m) {
                    const f2 *pp = sp + gq * 32 + ((lane + m) & 31);
                    f2 P[9];
#pragma unroll
                    for (int a = 0; a < 9; ++a) P[a] = pp[a * S];
                    f2 TM[3], TG[3];   // both targets' terms for the packet
                    vjp_sym_f32x2<TENSOR, PER, true>(XI[0], YI[0], ZI[0], FI[0], WI[0], P[0], P[1], P[2], P[3], P[4],
                                                     P[5], P[6], P[7], P[8], c, M[0], G[0], TM, TG);
#pragma unroll
                    for (int k = 1; k < R; ++k)
                        vjp_sym_f32x2<TENSOR, PER, false>(XI[k], YI[k], ZI[k], FI[k], WI[k], P[0], P[1], P[2], P[3],
                                                          P[4], P[5], P[6], P[7], P[8], c, M[k], G[k], TM, TG);
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        JM[d] = __shfl_sync(0xffffffffu, add2(JM[d], TM[d]), nxt);
                        JG[d] = __shfl_sync(0xffffffffu, sub2(JG[d], TG[d]), nxt);
                    }
                }
                fold();   // (32 terms per packed lane)
                for (int d = 0; d < 3; ++d) {   // lane holds packet `lane` of the group again
                    jw[d * S + gq * 32 + lane] = JM[d];
                    jw[(3 + d) * S + gq * 32 + lane] = JG[d];
                }
            }
        }
        if (diag) fold();
        __syncthreads();   // stage st consumed; every warp's source sums are in s_jacc
        if (!diag) {
            float *dst = jpart + static_cast<size_t>(t) * 6 * B;
            for (int e = tid; e < 6 * B; e += NT) {
                float v = s_jacc[e];
#pragma unroll
                for (int w = 1; w < NW; ++w) v = __fadd_rn(v, s_jacc[w * 6 * B + e]);
                dst[e] = v;
            }
            __syncthreads();   // s_jacc free for the next tile
        }
        aborted = s_abort != 0;
        if (tid == 0 && !aborted && t + 2 < t1) issue(st);
        if (++jb == g.nIB) { ++ib; jb = ib; }
    }
    flush(cur_ib);
    if (tid == 0) {
        for (int k = waited0; k < issued0; ++k)
            if (!mbar_wait_bounded(&bars[0], k & 1, drain_limit(wd))) atomicOr(err, DEV_ERR_TIMEOUT);
        for (int k = waited1; k < issued1; ++k)
            if (!mbar_wait_bounded(&bars[1], k & 1, drain_limit(wd))) atomicOr(err, DEV_ERR_TIMEOUT);
    }
}

// FP64, bound by the FP64 pipe (two operations a clock and SM): 77 operations an unordered
// pair.  One target per lane; blocks of 32 or 64 particles while there are few, so that the
// tiles reach every SM.  The sums are divided by c1.  Whole call at
// N = 200 / 1,500 / 4,096: 397 / 751 / 2,484 us directed, so 112 / 233 / 1,221; since the even
// spread counts the static arrays, a call waited for takes 224 us at 1,500 (256) and 371 at 2,000 (399).
template <int TENSOR, bool PER, int B>
__global__ void __launch_bounds__(B) vjp_sym64_kernel(const dbl4 *__restrict__ pos, const dbl4 *__restrict__ frc,
                                                      const dbl4 *__restrict__ wv, double *__restrict__ partM,
                                                      double *__restrict__ partG, double *__restrict__ jpart, int npad,
                                                      DenseGeom g, PairConst c) {
    constexpr int NW = B / 32;
    __shared__ double s_src[9][B];
    __shared__ double s_jacc[NW][6][B];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long t0 = static_cast<long long>(blockIdx.x) * g.chunk;
    const long long t1 = (t0 + g.chunk < g.nT) ? t0 + g.chunk : g.nT;
    if (t0 >= t1) return;
    int ib, jb, cur_ib = -1;
    sym_tile_at(g, t0, ib, jb);
    double T[9], M[3], G[3];
    auto flush = [&](int row) {
        const size_t at = static_cast<size_t>(blockIdx.x - geom_first(g, row)) * 3 * npad + static_cast<size_t>(row) * B + tid;
        for (int d = 0; d < 3; ++d) {
            partM[at + d * static_cast<size_t>(npad)] = M[d];
            partG[at + d * static_cast<size_t>(npad)] = G[d];
        }
    };
    auto load = [&](int block, double (&v)[9]) {
        const size_t i = static_cast<size_t>(block) * B + tid;
        const dbl4 p = pos[i], f = frc[i], w = wv[i];
        v[0] = p.x; v[1] = p.y; v[2] = p.z;
        v[3] = f.x; v[4] = f.y; v[5] = f.z;
        v[6] = w.x; v[7] = w.y; v[8] = w.z;
    };
    for (long long t = t0; t < t1; ++t) {
        if (ib != cur_ib) {
            if (cur_ib >= 0) flush(cur_ib);
            cur_ib = ib;
            load(ib, T);
            for (int d = 0; d < 3; ++d) M[d] = G[d] = 0.0;
        }
        {
            double v[9];
            load(jb, v);
            for (int d = 0; d < 9; ++d) s_src[d][tid] = v[d];
        }
        __syncthreads();
        const bool diag = ib == jb;
        if (diag) {
#pragma unroll 2
            for (int jj = 0; jj < B; ++jj) {
                double v[9];
                for (int d = 0; d < 9; ++d) v[d] = s_src[d][jj];
                vjp_sym_f64<TENSOR, PER, false>(T, v, c, M, G, M, G);
            }
        } else {
            const int nxt = (lane + 1) & 31;
#pragma unroll 1
            for (int gq = 0; gq < NW; ++gq) {
                double JM[3] = {0.0, 0.0, 0.0}, JG[3] = {0.0, 0.0, 0.0};
#pragma unroll 2
                for (int m = 0; m < 32; ++m) {
                    double v[9];
#pragma unroll
                    for (int d = 0; d < 9; ++d) v[d] = s_src[d][gq * 32 + ((lane + m) & 31)];
                    vjp_sym_f64<TENSOR, PER>(T, v, c, M, G, JM, JG);
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        JM[d] = __shfl_sync(0xffffffffu, JM[d], nxt);
                        JG[d] = __shfl_sync(0xffffffffu, JG[d], nxt);
                    }
                }
                for (int d = 0; d < 3; ++d) {
                    s_jacc[warp][d][gq * 32 + lane] = JM[d];
                    s_jacc[warp][3 + d][gq * 32 + lane] = JG[d];
                }
            }
        }
        __syncthreads();
        if (!diag) {
            double *dst = jpart + static_cast<size_t>(t) * 6 * B;
            for (int e = tid; e < 6 * B; e += B) {
                double v = s_jacc[0][e / B][tid];
#pragma unroll
                for (int w = 1; w < NW; ++w) v += s_jacc[w][e / B][tid];
                dst[e] = v;
            }
        }
        // (the next tile's writes of s_jacc come after its first barrier)
        if (++jb == g.nIB) { ++ib; jb = ib; }
    }
    flush(cur_ib);
}

// Above this the directed kernels (the source-side sums of the block pairs are 202 MB here in FP32C,
// 807 MB in FP64).
constexpr int kVjpSymN = 65536;

// Dynamic shared memory: FP64, two stages of three dbl4 arrays; FP32C, two stages of
// nine float arrays and the (hi, lo) accumulators, and (symmetric) the warps' source sums.
static size_t vjp_smem(int mode, int J) {
    if (mode == MODE_FP64) return 6 * static_cast<size_t>(J) * sizeof(dbl4);
    return 18 * static_cast<size_t>(J) * sizeof(float) + static_cast<size_t>(kRV2) * 12 * kNT * sizeof(float);
}
constexpr size_t vjp_sym_smem(int B, int NT) { return (18 + 12 + 6 * (NT / 32)) * static_cast<size_t>(B) * sizeof(float); }

using Vjp2Fn = void (*)(const float *, const float *, const float *, double *, double *, int, DenseGeom, VjpConst2, int *,
                        long long);
using Vjp64Fn = void (*)(const dbl4 *, const dbl4 *, const dbl4 *, double *, double *, int, DenseGeom, PairConst, int *,
                         long long);
using VjpSymFn = void (*)(const float *, const float *, const float *, double *, double *, float *, int, DenseGeom,
                          VjpConst2, int *, long long);
using VjpSym64Fn = void (*)(const dbl4 *, const dbl4 *, const dbl4 *, double *, double *, double *, int, DenseGeom,
                            PairConst);
#define SD_VJP_PICK(FN, ...)                                                                                  \
    (h->tensor == T_OSEEN ? (h->pc.periodic ? FN<T_OSEEN, true, ##__VA_ARGS__> : FN<T_OSEEN, false, ##__VA_ARGS__>) \
                          : (h->pc.periodic ? FN<T_RP, true, ##__VA_ARGS__> : FN<T_RP, false, ##__VA_ARGS__>))
static Vjp2Fn pick_vjp2(const sd_handle *h) { return SD_VJP_PICK(vjp2_kernel); }
static Vjp64Fn pick_vjp64(const sd_handle *h) { return SD_VJP_PICK(vjp_kernel); }
static VjpSymFn pick_vjp_sym(const sd_handle *h, int B) {
    if (B == 64) return SD_VJP_PICK(vjp_sym_kernel, 64, 32);
    if (B == 128) return SD_VJP_PICK(vjp_sym_kernel, 128, 64);
    return SD_VJP_PICK(vjp_sym_kernel, 256, 128);
}
static VjpSym64Fn pick_vjp_sym64(const sd_handle *h, int B) {
    if (B == 32) return SD_VJP_PICK(vjp_sym64_kernel, 32);
    if (B == 64) return SD_VJP_PICK(vjp_sym64_kernel, 64);
    return SD_VJP_PICK(vjp_sym64_kernel, 128);
}
#undef SD_VJP_PICK

// The grid holds SD_VJP_CTA_SCALE times as many CTAs as fit at once, so the block
// scheduler evens out the SMs' shares (directed kernel, N = 4,096: 57 -> 51 us; 8x gave the
// same); the symmetric kernels take a tile per CTA, or runs once there are many (dense_setup).
#ifndef SD_VJP_CTA_SCALE
#define SD_VJP_CTA_SCALE 2
#endif
#ifndef SD_VJP_JMIN
#define SD_VJP_JMIN 64   // smallest j-tile (32 measured slower at N = 4,096)
#endif
cudaError_t vjp_setup(sd_handle *h) {
    DenseGeom g{};
    const int mode = (h->mode == MODE_FP64) ? MODE_FP64 : MODE_FP32C;
    int occ = 0;
    if (h->n <= kVjpSymN) {
        // blocks: FP64 32 / 64 / 128 particles, FP32C 64 / 128 / 256, larger ones (fewer
        // source-side rows) once their tiles are 12 per SM, the FP32C ones of 128 (two warps
        // per CTA) from 3 on (N = 4,096, whole call: 76 us with 128, 80 with 64; 8,192: 143 with
        // 128, 153 with 256)
        const int unit = mode == MODE_FP64 ? 32 : 64;
        int B = unit;
        for (; B < 4 * unit; B *= 2) {
            const long long nb = (h->n + 2 * B - 1) / (2 * B);
            if (nb * (nb + 1) / 2 < (B == 64 && unit == 64 ? 3LL : 12LL) * h->num_sms) break;
        }
        g.sym = 1;
        g.I = g.J = B;
        g.nIB = g.nJT = (std::max(h->n, 1) + B - 1) / B;
        g.nT = static_cast<long long>(g.nIB) * (g.nIB + 1) / 2;
        const void *fn = mode == MODE_FP64 ? reinterpret_cast<const void *>(pick_vjp_sym64(h, B))
                                           : reinterpret_cast<const void *>(pick_vjp_sym(h, B));
        cudaError_t e = allow_smem(fn, h->vjp_limit);
        if (e == cudaSuccess)
            e = mode == MODE_FP64 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, B, 0)
                                  : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, B / 2, vjp_sym_smem(B, B / 2));
        if (e != cudaSuccess) return e;
        occ = std::max(occ, 1);
        const long long resident = static_cast<long long>(h->num_sms) * occ;
        g.chunk = g.nT <= 32 * resident ? 1 : (g.nT + 16 * resident - 1) / (16 * resident);
    } else {
        g.I = kNT * (mode == MODE_FP64 ? kRV : kRV2);
        g.nIB = h->npad / g.I;
        const void *fn = mode == MODE_FP64 ? reinterpret_cast<const void *>(pick_vjp64(h))
                                           : reinterpret_cast<const void *>(pick_vjp2(h));
        cudaError_t e = allow_smem(fn, h->vjp_limit);
        if (e != cudaSuccess) return e;
        const int Jc[4] = {kJmax, 128, 64, SD_VJP_JMIN};
        for (int ci = 0; ci < 4; ++ci) {
            const int J = Jc[ci];
            if (mode == MODE_FP64 && J > 128) continue;
            const size_t smem = vjp_smem(mode, J);
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kNT, smem);
            if (e != cudaSuccess) return e;
            g.J = J;
            g.nJT = h->npad / J;
            if (static_cast<long long>(g.nIB) * g.nJT >= 4LL * h->num_sms * std::max(occ, 1)) break;
        }
        occ = std::max(occ, 1);
        g.nT = static_cast<long long>(g.nIB) * g.nJT;
        const long long want = static_cast<long long>(h->num_sms) * occ * SD_VJP_CTA_SCALE;
        g.chunk = std::max(1LL, (g.nT + want - 1) / want);
    }
    g.grid = static_cast<int>((g.nT + g.chunk - 1) / g.chunk);
    int ms = 0;
    for (int ib = 0; ib < g.nIB; ++ib) ms = std::max(ms, geom_last(g, ib) - geom_first(g, ib) + 1);
    g.maxSlots = ms;
    h->geomv = g;
    h->vjp_occ = occ;
    return cudaSuccess;
}

static VjpConst2 vjp_const2(const PairConst &pc) {
    VjpConst2 c{};
    c.c1 = pk2_host(pc.c1_f);
    c.c3 = pk2_host(pc.c3_f);
    c.m3c3 = pk2_host(pc.m3c3_f);
    c.nc1 = pk2_host(-pc.c1_f);
    c.n5m3c3 = pk2_host(-5.0f * pc.m3c3_f);
    c.n3c1 = pk2_host(-3.0f * pc.c1_f);
    c.r2min = pc.r2min_f;
    for (int d = 0; d < 3; ++d) {
        c.negL[d] = pk2_host(-pc.Lf[d]);
        c.invL[d] = pk2_host(pc.invLf[d]);
    }
    return c;
}

cudaError_t launch_vjp_dense(sd_handle *h, cudaStream_t st, Mirror posm, Mirror frcm, Mirror wm) {
    const DenseGeom &g = h->geomv;
    double *partM = h->vpartM, *partG = h->vpartG;
    const bool f64 = h->mode == MODE_FP64;
    const size_t sym_smem =
        g.sym ? spread_smem(h->num_sms, g.grid, h->vjp_occ, f64 ? 0 : vjp_sym_smem(g.I, g.I / 2), h->vjp_limit) : 0;
    prof_begin(h, SD_KERNEL_VJP, st);
    if (f64) {
        const dbl4 *p = static_cast<const dbl4 *>(posm.aos), *f = static_cast<const dbl4 *>(frcm.aos),
                   *w = static_cast<const dbl4 *>(wm.aos);
        if (g.sym)
            pick_vjp_sym64(h, g.I)<<<g.grid, g.I, sym_smem, st>>>(p, f, w, partM, partG, static_cast<double *>(h->vjpart), h->npad,
                                                          g, h->pc);
        else
            pick_vjp64(h)<<<g.grid, kNT, vjp_smem(MODE_FP64, g.J), st>>>(p, f, w, partM, partG, h->npad, g, h->pc,
                                                                       h->d_err, h->watchdog);
    } else {
        const VjpConst2 c = vjp_const2(h->pc);
        if (g.sym)
            pick_vjp_sym(h, g.I)<<<g.grid, g.I / 2, sym_smem, st>>>(
                posm.soa, frcm.soa, wm.soa, partM, partG, static_cast<float *>(h->vjpart), h->npad, g, c, h->d_err,
                h->watchdog);
        else
            pick_vjp2(h)<<<g.grid, kNT, vjp_smem(MODE_FP32C, g.J), st>>>(posm.soa, frcm.soa, wm.soa, partM, partG,
                                                                       h->npad, g, c, h->d_err, h->watchdog);
    }
    prof_end(h, SD_KERNEL_VJP, st);
    ++h->launches;
    return cudaGetLastError();
}

// ---------------------------------------------------------------- near pairs and epilogue

struct VjpEpiArgs {
    const double *partM, *partG;
    const void *jpart;       // source-side sums of the symmetric kernels (g.sym)
    int npad;
    DenseGeom g;
    const double *x64;
    const void *posm;
    const double *F64;
    const void *frcm;
    const double *W64;
    void *wm;                // the cotangents' mirror (adjoint: rewritten for the next step)
    float *wsoa;
    CellList cl;
    double rnear2;
    PairConst pc;
    VjpConst2 c2;
    int n;
    // candidate list of the near pass or the Verlet steps, and its pairs' terms
    const int2 *ent;
    double *ent_out;         // [cap][6]: mu W (3), x gradient (3), exact minus all-pairs term
    const unsigned long long *ent_n;
    const int *noff, *ncnt;  // (-1: in near[i])
    int cap;
    double *near;            // [n][6]
    int out_dtype;   // SD_DTYPE_F32 / SD_DTYPE_F64 for gX / gF, or -1 = adjoint update
    void *gx_out, *gF_out;
    double dt;
    double *lam_out;   // adjoint: lam_out = W + dt gX
    double *gF_acc;    // adjoint: gF_acc += dt mu W
    int *err;
};

// What the all-pairs kernel adds to the target i's sums for the pair (i, j), i in block bi and
// j in block bj of its tiling: the same operations on the same operands (FP32C), taken from
// the side on which the tile has them.
template <int TENSOR, int MODE, bool PER>
__device__ __forceinline__ void vjp_dense_term(const VjpEpiArgs &a, int i, int j, double (&o)[6]) {
    constexpr int TD = (TENSOR == T_OSEEN) ? T_OSEEN : T_RP;
    using V4 = typename VjpT<MODE>::V4;
    const V4 *pm = static_cast<const V4 *>(a.posm), *fm = static_cast<const V4 *>(a.frcm),
             *wm = static_cast<const V4 *>(a.wm);
    const int bi = i / a.g.I, bj = j / a.g.I;
    const bool swap = a.g.sym && bi > bj;   // the tile has j's block as its targets
    const int t = swap ? j : i, s = swap ? i : j;
    const V4 pt = pm[t], ft = fm[t], wt = wm[t], ps = pm[s], fs = fm[s], ws = wm[s];
    if constexpr (MODE == MODE_FP64) {
        const double vt[9] = {pt.x, pt.y, pt.z, ft.x, ft.y, ft.z, wt.x, wt.y, wt.z};
        const double vs[9] = {ps.x, ps.y, ps.z, fs.x, fs.y, fs.z, ws.x, ws.y, ws.z};
        double M[3] = {}, G[3] = {}, JM[3] = {}, JG[3] = {};
        vjp_sym_f64<TD, PER>(vt, vs, a.pc, M, G, JM, JG);
        for (int d = 0; d < 3; ++d) {
            o[d] = a.pc.c1_d * (swap ? JM[d] : M[d]);
            o[3 + d] = a.pc.c1_d * (swap ? JG[d] : G[d]);
        }
    } else {
        f2 M[3] = {}, G[3] = {}, JM[3] = {}, JG[3] = {};
        auto two = [](float v) { return pk2(v, v); };
        const f2 FI[3] = {two(ft.x), two(ft.y), two(ft.z)}, WI[3] = {two(wt.x), two(wt.y), two(wt.z)};
        if (a.g.sym && bi != bj)
            vjp_sym_f32x2<TD, PER, true>(two(pt.x), two(pt.y), two(pt.z), FI, WI, two(ps.x), two(ps.y), two(ps.z), two(fs.x),
                                         two(fs.y), two(fs.z), two(ws.x), two(ws.y), two(ws.z), a.c2, M, G, JM, JG);
        else
            vjp_pair_f32x2<TD, PER>(two(pt.x), two(pt.y), two(pt.z), FI[0], FI[1], FI[2], WI[0], WI[1], WI[2], two(ps.x),
                                    two(ps.y), two(ps.z), two(fs.x), two(fs.y), two(fs.z), two(ws.x), two(ws.y),
                                    two(ws.z), a.c2, M, G);
        for (int d = 0; d < 3; ++d) {
            float lo, hi;
            upk2(swap ? JM[d] : M[d], lo, hi);
            o[d] = static_cast<double>(lo);
            upk2(swap ? JG[d] : G[d], lo, hi);
            o[3 + d] = swap ? -static_cast<double>(lo) : static_cast<double>(lo);
        }
    }
}

// The pair (i, j) if it is closer than r_near: the exact FP64 terms minus the all-pairs
// kernel's, added to o.
template <int TENSOR, int MODE>
__device__ __forceinline__ void vjp_near_term(const VjpEpiArgs &a, int i, int j, double (&o)[6], bool &coincident) {
    double dx = a.x64[3 * i] - a.x64[3 * j], dy = a.x64[3 * i + 1] - a.x64[3 * j + 1],
           dz = a.x64[3 * i + 2] - a.x64[3 * j + 2];
    box_image(a.cl.box, dx, dy, dz);
    const double r2 = dx * dx + dy * dy + dz * dz;
    if (r2 >= a.rnear2) return;
    if (r2 == 0.0 && TENSOR != T_RPY) {
        coincident = true;
        return;
    }
    double A, B, dA, dB;
    profile_exact<TENSOR>(r2, a.pc, A, B, dA, dB);
    const double Fx = a.F64[3 * i], Fy = a.F64[3 * i + 1], Fz = a.F64[3 * i + 2];
    const double Wx = a.W64[3 * i], Wy = a.W64[3 * i + 1], Wz = a.W64[3 * i + 2];
    const double fx = a.F64[3 * j], fy = a.F64[3 * j + 1], fz = a.F64[3 * j + 2];
    const double wx = a.W64[3 * j], wy = a.W64[3 * j + 1], wz = a.W64[3 * j + 2];
    const double Wir = dx * Wx + dy * Wy + dz * Wz, Fir = dx * Fx + dy * Fy + dz * Fz;
    const double Wjr = dx * wx + dy * wy + dz * wz, Fjr = dx * fx + dy * fy + dz * fz;
    const double U = Wx * fx + Wy * fy + Wz * fz + wx * Fx + wy * Fy + wz * Fz;
    const double Q = Wir * Fjr + Wjr * Fir;
    const double cr = dA * U + dB * Q;
    double t[6];
    if (a.pc.periodic) vjp_dense_term<TENSOR, MODE, true>(a, i, j, t);
    else vjp_dense_term<TENSOR, MODE, false>(a, i, j, t);
    o[0] += A * wx + B * Wjr * dx - t[0];
    o[1] += A * wy + B * Wjr * dy - t[1];
    o[2] += A * wz + B * Wjr * dz - t[2];
    o[3] += cr * dx + B * (Wx * Fjr + fx * Wir + wx * Fir + Fx * Wjr) - t[3];
    o[4] += cr * dy + B * (Wy * Fjr + fy * Wir + wy * Fir + Fy * Wjr) - t[4];
    o[5] += cr * dz + B * (Wz * Fjr + fz * Wir + wz * Fir + Fz * Wjr) - t[5];
}

// One thread per listed pair, so that the FP64 operations (some 150 a pair, two a clock and
// SM) run with full warps; then the particles that a full list left out.  A walk over the
// cells inside the epilogue took 45 us at N = 4,096, nearly all of it in warps with one or
// two pairs; this kernel takes 9 us, beside the all-pairs kernel in the adjoint, and the
// epilogue 10.
template <int TENSOR, int MODE>
__global__ void __launch_bounds__(64) vjp_near_kernel(VjpEpiArgs a) {
    const long long gt = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x,
                    stride = static_cast<long long>(gridDim.x) * blockDim.x;
    const long long total = static_cast<long long>(min(*a.ent_n, static_cast<unsigned long long>(a.cap)));
    bool coincident = false;
    for (long long e = gt; e < total; e += stride) {
        const int2 p = a.ent[e];
        double o[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        if (p.x >= 0)
            vjp_near_term<TENSOR, MODE>(a, static_cast<int>(dbg_index(p.x, a.n, a.err)),
                                        static_cast<int>(dbg_index(p.y, a.n, a.err)), o, coincident);
        for (int d = 0; d < 6; ++d) a.ent_out[6 * e + d] = o[d];
    }
    if (*a.ent_n > static_cast<unsigned long long>(a.cap))
        for (long long i = gt; i < a.n; i += stride) {
            if (a.ncnt[i] >= 0) continue;
            double o[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
            for_each_neighbour_part(a.cl, static_cast<int>(i), a.cl.cell[i], 0, 1, [&](int j) {
                vjp_near_term<TENSOR, MODE>(a, static_cast<int>(i), j, o, coincident);
            });
            for (int d = 0; d < 6; ++d) a.near[6 * i + d] = o[d];
        }
    if (coincident) atomicOr(a.err, DEV_ERR_COINCIDENT);
}

// 32 particles per CTA: its warps add the slots and the source-side rows of the particles'
// block column in turn (lane = particle), warp 0 adds the warps' sums in ascending order and
// finishes (the shape of epilogue_kernel).
constexpr int kVjpEpiWarps = 8;
template <int TENSOR, int MODE>
__global__ void __launch_bounds__(32 * kVjpEpiWarps) vjp_epilogue_kernel(VjpEpiArgs a) {
    using V4 = typename VjpT<MODE>::V4;
    constexpr int W = kVjpEpiWarps;
    constexpr bool F64 = MODE == MODE_FP64;
    __shared__ float2 s_f[F64 ? 1 : W][6][32];
    __shared__ double s_d[F64 ? W : 1][6][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = (gridDim.x - 1 - blockIdx.x) * 32 + lane;   // (the longest columns first)
    const bool active = i < a.n;
    int off = 0, cnt = 0;
    V4 wi{};
    double Wd[3] = {0.0, 0.0, 0.0}, acc[3] = {0.0, 0.0, 0.0};
    if (w == 0 && active) {   // needed last, asked for first
        off = a.noff[i];
        cnt = a.ncnt[i];
        wi = static_cast<const V4 *>(a.wm)[i];
        for (int d = 0; d < 3; ++d) {
            Wd[d] = a.W64[3 * i + d];
            if (a.out_dtype < 0) acc[d] = a.gF_acc[3 * i + d];
        }
    }
    if (active) {
        const int ib = i / a.g.I, ns = geom_last(a.g, ib) - geom_first(a.g, ib) + 1, nc = a.g.sym ? ib : 0;
        const int o = i - ib * a.g.I, J = a.g.J;
        const size_t np = a.npad, cs = 6 * static_cast<size_t>(J);
        if constexpr (F64) {
            const double *jp = static_cast<const double *>(a.jpart);
            double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
            for (int s = w; s < ns; s += W)
                for (int d = 0; d < 3; ++d) {
                    v[d] += a.partM[(static_cast<size_t>(s) * 3 + d) * np + i];
                    v[3 + d] += a.partG[(static_cast<size_t>(s) * 3 + d) * np + i];
                }
            for (int r = w; r < nc; r += W) {
                const double *src = jp + static_cast<size_t>(geom_rowstart(a.g, r) + (ib - r)) * cs + o;
                for (int d = 0; d < 6; ++d) v[d] += src[d * J];
            }
            for (int d = 0; d < 6; ++d) s_d[w][d][lane] = v[d];
        } else {   // (hi, lo) float pairs, summed with FP32 TwoSum (FP64 issues at 1/64 the rate)
            const float2 *pM = reinterpret_cast<const float2 *>(a.partM), *pG = reinterpret_cast<const float2 *>(a.partG);
            const float *jp = static_cast<const float *>(a.jpart);
            float hi[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, lo[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 2
            for (int s = w; s < ns; s += W)
                for (int d = 0; d < 6; ++d) {
                    const float2 q = (d < 3 ? pM : pG)[(static_cast<size_t>(s) * 3 + d % 3) * np + i];
                    fold2(hi[d], lo[d], q.x);
                    lo[d] = __fadd_rn(lo[d], q.y);
                }
#pragma unroll 2
            for (int r = w; r < nc; r += W) {
                const float *src = jp + static_cast<size_t>(geom_rowstart(a.g, r) + (ib - r)) * cs + o;
                for (int d = 0; d < 6; ++d) fold2(hi[d], lo[d], src[d * J]);
            }
            for (int d = 0; d < 6; ++d) s_f[w][d][lane] = make_float2(hi[d], lo[d]);
        }
    }
    __syncthreads();
    if (w != 0 || !active) return;
    double MG[6];
    for (int d = 0; d < 6; ++d) {
        if constexpr (F64) {
            double v = s_d[0][d][lane];
            for (int q = 1; q < W; ++q) v += s_d[q][d][lane];
            MG[d] = a.pc.c1_d * v;
        } else {
            float h = s_f[0][d][lane].x, l = s_f[0][d][lane].y;
            for (int q = 1; q < W; ++q) {
                fold2(h, l, s_f[q][d][lane].x);
                l = __fadd_rn(l, s_f[q][d][lane].y);
            }
            MG[d] = static_cast<double>(h) + static_cast<double>(l);
        }
    }
    {   // self: mu_ii W_i / mu0 = W_i instead of the clamped term; its x-derivative is zero
        double A;
        if constexpr (F64) {
            double Ad, Bd;
            profile64<(TENSOR == T_OSEEN) ? T_OSEEN : T_RP>(a.pc.r2min_d, a.pc, Ad, Bd);
            A = a.pc.c1_d * Ad;
            MG[0] += Wd[0] - A * wi.x;
            MG[1] += Wd[1] - A * wi.y;
            MG[2] += Wd[2] - A * wi.z;
        } else {
            const float ri = rsqrt_sfu(a.pc.r2min_f), ri2 = __fmul_rn(ri, ri);
            const float Af = TENSOR == T_OSEEN ? __fmul_rn(a.pc.c1_f, ri)
                                               : __fmul_rn(ri, __fmaf_rn(a.pc.c3_f, ri2, a.pc.c1_f));
            MG[0] += Wd[0] - static_cast<double>(__fmul_rn(Af, wi.x));
            MG[1] += Wd[1] - static_cast<double>(__fmul_rn(Af, wi.y));
            MG[2] += Wd[2] - static_cast<double>(__fmul_rn(Af, wi.z));
        }
    }
    if (cnt < 0) {
        for (int d = 0; d < 6; ++d) MG[d] += a.near[6 * static_cast<size_t>(i) + d];
    } else {
        const double *e = a.ent_out + 6 * static_cast<size_t>(dbg_index(off, static_cast<long long>(a.cap) - cnt + 1, a.err));
        for (int k = 0; k < cnt; ++k, e += 6)
            for (int d = 0; d < 6; ++d) MG[d] += e[d];
    }
    const double m0 = a.pc.mu0;
    if (a.out_dtype == SD_DTYPE_F32) {
        float *gx = static_cast<float *>(a.gx_out), *gF = static_cast<float *>(a.gF_out);
        for (int d = 0; d < 3; ++d) {
            if (gx) gx[3 * i + d] = static_cast<float>(m0 * MG[3 + d]);
            if (gF) gF[3 * i + d] = static_cast<float>(m0 * MG[d]);
        }
    } else if (a.out_dtype == SD_DTYPE_F64) {
        double *gx = static_cast<double *>(a.gx_out), *gF = static_cast<double *>(a.gF_out);
        for (int d = 0; d < 3; ++d) {
            if (gx) gx[3 * i + d] = m0 * MG[3 + d];
            if (gF) gF[3 * i + d] = m0 * MG[d];
        }
    } else {   // lambda, the cotangents of the next step back, and their mirror
        double l[3];
        for (int d = 0; d < 3; ++d) {
            l[d] = Wd[d] + a.dt * (m0 * MG[3 + d]);
            a.lam_out[3 * i + d] = l[d];
            a.gF_acc[3 * i + d] = acc[d] + a.dt * (m0 * MG[d]);
        }
        if (!isfinite(l[0]) || !isfinite(l[1]) || !isfinite(l[2])) atomicOr(a.err, DEV_ERR_NONFINITE);
        put_mirror(static_cast<V4 *>(a.wm), a.wsoa, a.npad, i, l[0], l[1], l[2]);
    }
}

static VjpEpiArgs vjp_epi_args(sd_handle *h, const VjpInput &in) {
    VjpEpiArgs a{};
    a.partM = h->vpartM;
    a.partG = h->vpartG;
    a.jpart = h->vjpart;
    a.npad = h->npad;
    a.g = h->geomv;
    a.x64 = in.x64;
    a.posm = h->posm.aos;
    a.F64 = in.F64;
    a.frcm = in.frcm.aos;
    a.W64 = in.W64;
    a.wm = h->wam.aos;
    a.wsoa = h->wam.soa;
    a.cl = h->cl;
    a.rnear2 = h->r_near * h->r_near;
    a.pc = h->pc;
    a.c2 = vjp_const2(h->pc);
    a.n = h->n;
    a.ent = in.vlist ? h->vent : h->near_ent;
    a.ent_out = h->near_out;
    a.ent_n = in.vlist ? h->vn : h->near_n;
    a.noff = in.vlist ? h->voff : h->near_off;
    a.ncnt = in.vlist ? h->vcnt : h->near_cnt;
    a.cap = h->near_cap;
    a.near = h->near64;
    a.err = h->d_err;
    return a;
}

#define SD_VJP_DISPATCH(FN, NB, NTH)                                                                             \
    do {                                                                                                         \
        const bool f64_ = h->mode == MODE_FP64;                                                                  \
        switch (h->tensor) {                                                                                     \
            case T_RPY:                                                                                          \
                if (f64_) FN<T_RPY, MODE_FP64><<<NB, NTH, 0, st>>>(a);                                           \
                else FN<T_RPY, MODE_FP32C><<<NB, NTH, 0, st>>>(a);                                               \
                break;                                                                                           \
            case T_RP:                                                                                           \
                if (f64_) FN<T_RP, MODE_FP64><<<NB, NTH, 0, st>>>(a);                                            \
                else FN<T_RP, MODE_FP32C><<<NB, NTH, 0, st>>>(a);                                                \
                break;                                                                                           \
            default:                                                                                             \
                if (f64_) FN<T_OSEEN, MODE_FP64><<<NB, NTH, 0, st>>>(a);                                         \
                else FN<T_OSEEN, MODE_FP32C><<<NB, NTH, 0, st>>>(a);                                             \
                break;                                                                                           \
        }                                                                                                        \
    } while (0)

cudaError_t launch_vjp_near(sd_handle *h, cudaStream_t st, const VjpInput &in) {
    if (h->n == 0) return cudaSuccess;
    const VjpEpiArgs a = vjp_epi_args(h, in);
    const int nb = static_cast<int>(std::min<long long>((static_cast<long long>(h->n) * 4 + 63) / 64, 8LL * h->num_sms));
    SD_VJP_DISPATCH(vjp_near_kernel, nb, 64);
    ++h->launches;
    return cudaGetLastError();
}

cudaError_t launch_vjp_epilogue(sd_handle *h, cudaStream_t st, const VjpInput &in, int out_dtype, void *gx_out,
                                void *gF_out, double dt, double *lam_out, double *gF_acc) {
    if (h->n == 0) return cudaSuccess;
    VjpEpiArgs a = vjp_epi_args(h, in);
    a.out_dtype = out_dtype;
    a.gx_out = gx_out;
    a.gF_out = gF_out;
    a.dt = dt;
    a.lam_out = lam_out;
    a.gF_acc = gF_acc;
    prof_begin(h, SD_KERNEL_EPILOGUE, st);
    SD_VJP_DISPATCH(vjp_epilogue_kernel, (h->n + 31) / 32, 32 * kVjpEpiWarps);
    prof_end(h, SD_KERNEL_EPILOGUE, st);
    ++h->launches;
    return cudaGetLastError();
}
#undef SD_VJP_DISPATCH

}  // namespace sd
