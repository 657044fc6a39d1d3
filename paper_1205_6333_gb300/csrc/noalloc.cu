// noalloc.cu -- sd_mobility_apply_noalloc: the mobility product v = mu(x) F for
// callers that must not allocate GPU memory.
//
// Who needs it: code that runs while a CUDA stream is being captured into a
// graph (cudaMalloc cannot be captured and a graph replay could not repeat it),
// hosts that hand a plug-in a fixed device-memory budget and forbid further
// allocation, and latency-critical loops that cannot afford cudaMalloc/cudaFree
// (which may synchronise the device).  Such a caller cannot create an sd_handle,
// because a handle allocates its buffers.
//
// This entry point allocates nothing.  Its only working memory (FP32 copies of
// the inputs and the per-split partial sums of the all-pairs kernel) lives in
// one file-scope __device__ array of kScratchBytes (about 14 MB), which every
// GPU that loads the library holds until the process exits.  That array bounds
// the problem size to n <= kMaxN (65,536 particles).
//
// The kernels here are a self-contained variant of the all-pairs sum of
// dense.cu: FP32 pair terms with compensated (two-float) accumulation, the
// (target block, source tile) plane cut into equal runs over the CTAs with
// partial sums in the scratch array, the self term and overlapping pairs handled
// exactly inside the pair loop (so no cell list and no FP64 near-pair pass are
// needed), and a final FP64 reduction.
//
// What bounds it is the FP32 pipe.  Two sources share every instruction (the packed
// f32x2 operations), a thread owns two targets so that a load serves four pairs, and a
// group of pairs leaves the packed path only where one of them is closer than 2a, so
// nothing is clamped.  Every pair is evaluated in both directions: using it once, as
// dense_sym_kernel does, needs the source-side sums of every tile beside the target sums,
// 50 MB at n = 65,536 with blocks of 512, where the scratch array has 12 MB.  (Up to about
// 20,000 particles both would fit, 5 + 6 MB; that form is not built.)  Whole call at n = 3,000 / 20,011 / 65,536 with scalar
// pair terms, one target per thread and eight splits whatever n is: 55 / 570 / 4,844 us;
// this way 39 / 367 / 3,300 us (22 FP32 operations per ordered pair: 67% of the pipe).
#include <cmath>
#include <mutex>
#include <string>

#include "sd_internal.h"

namespace sd {
namespace {

constexpr int kMaxN = 65536;          // largest n the scratch array holds
constexpr int kSplits = 8;            // partial sums per particle at n = kMaxN (more fit below)
constexpr int kThreads = 128;         // threads per CTA
constexpr int kTile = 256;            // largest j-tile, and what the scratch stride is rounded to
constexpr int kResident = 4;          // CTAs per SM the all-pairs kernel is compiled for (128 registers)
constexpr size_t kMirrorFloats = 6 * static_cast<size_t>(kMaxN);                  // x y z Fx Fy Fz (SoA)
constexpr size_t kPartialDoubles = static_cast<size_t>(kSplits) * 3 * kMaxN;       // [split][dim][i]
constexpr size_t kScratchBytes = kMirrorFloats * sizeof(float) + kPartialDoubles * sizeof(double);
constexpr int kMaxDevices = 64;

static_assert(kMaxN % kTile == 0, "the scratch stride must hold whole tiles");

// The scratch array.  Host code must not pass its name to a kernel: on the host
// the name is only a stand-in, so its device address is looked up once per
// device with cudaGetSymbolAddress (noalloc_scratch below).
__device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

std::mutex g_mutex;
void *g_scratch_ptr[kMaxDevices] = {};

// Device address of the scratch array on the current device (set up on the
// first call on each device), and the device's SMs.
int g_sms[kMaxDevices] = {};
sd_status noalloc_scratch(void **out, int *sms) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_status(e, "cudaGetDevice");
    if (dev < 0 || dev >= kMaxDevices) return set_error(SD_ERR_UNSUPPORTED, "device ordinal beyond 63");
    std::lock_guard<std::mutex> lock(g_mutex);
    if (!g_scratch_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) return cuda_status(e, "cudaGetSymbolAddress of the no-alloc scratch");
        e = cudaDeviceGetAttribute(&g_sms[dev], cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return cuda_status(e, "cudaDeviceGetAttribute");
        g_scratch_ptr[dev] = p;
    }
    *out = g_scratch_ptr[dev];
    *sms = g_sms[dev];
    return SD_OK;
}

struct NaArgs {
    const double *x, *F;
    double *V;
    int n, npad;       // npad: n rounded up to whole tiles, the stride of the scratch arrays
    DenseGeom g;       // target blocks, source tiles and the runs of tiles per CTA
    float *mir;        // scratch: SoA x, y, z, Fx, Fy, Fz with stride npad
    double *part;      // scratch: [slot][dim][npad]
    PairConst pc;
    PairConst2 c2;
};

// FP32 position (relative to particle 0) and force of particle i; past n far away, force-free.
__device__ __forceinline__ void na_load(const NaArgs &a, int i, float (&v)[6]) {
    v[0] = 1.0e18f;
    v[1] = v[2] = v[3] = v[4] = v[5] = 0.0f;
    if (i < a.n)
        for (int d = 0; d < 3; ++d) {
            v[d] = static_cast<float>(a.x[3 * i + d] - a.x[d]);
            v[3 + d] = static_cast<float>(a.F[3 * i + d]);
        }
}

// The mirror; entries n..npad-1 are rewritten on every call, since the array keeps whatever
// an earlier call left there.
__global__ void na_stage_kernel(NaArgs a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.npad) return;
    float v[6];
    na_load(a, i, v);
    for (int k = 0; k < 6; ++k) a.mir[k * static_cast<size_t>(a.npad) + i] = v[k];
}

// Exact pair term from zero (the overlap form for RPY when r < 2a), FP32.
template <int TENSOR>
__device__ __forceinline__ void na_exact(float dx, float dy, float dz, float fx, float fy, float fz,
                                         const PairConst &c, float &ax, float &ay, float &az) {
    const float r2 = dx * dx + dy * dy + dz * dz;
    if (r2 == 0.0f) {
        if (TENSOR == T_RPY) {   // coincident spheres: T^(0) = I
            ax += fx;
            ay += fy;
            az += fz;
        } else {                 // undefined for RP / Oseen: poison the result
            ax = ay = az = __int_as_float(0x7fc00000);
        }
        return;
    }
    const float r = sqrtf(r2);
    float A, B;
    if (TENSOR == T_RPY && r < static_cast<float>(c.two_a)) {
        A = 1.0f - 9.0f * r / (32.0f * static_cast<float>(c.a));
        B = 3.0f / (32.0f * static_cast<float>(c.a) * r);
    } else if (TENSOR == T_OSEEN) {
        A = c.c1_f / r;
        B = A / r2;
    } else {
        const float ri = 1.0f / r, ri2 = ri * ri;
        A = ri * (c.c1_f + c.c3_f * ri2);
        B = ri * ri2 * (c.c1_f + c.m3c3_f * ri2);
    }
    const float s = B * (dx * fx + dy * fy + dz * fz);
    ax += A * fx + s * dx;
    ay += A * fy + s * dy;
    az += A * fz + s * dz;
}

// The pairs of a group that holds one closer than 2a: each by its own r^2.
template <int TENSOR>
__device__ __noinline__ void na_group(float xi, float yi, float zi, const float *src, int J, int self, const PairConst &c,
                                      float (&o)[3]) {
    constexpr int TD = (TENSOR == T_OSEEN) ? T_OSEEN : T_RP;
    for (int u = 0; u < 4; ++u) {
        const float4 p = make_float4(src[u], src[J + u], src[2 * J + u], 0.0f);
        const float4 f = make_float4(src[3 * J + u], src[4 * J + u], src[5 * J + u], 0.0f);
        const float dx = xi - p.x, dy = yi - p.y, dz = zi - p.z;
        if (dx * dx + dy * dy + dz * dz >= c.r2min_f)
            pair_f32<TD, false>(xi, yi, zi, p, f, c, o[0], o[1], o[2]);
        else if (u != self)   // overlapping pair (rare); the self pair is skipped
            na_exact<TENSOR>(dx, dy, dz, f.x, f.y, f.z, c, o[0], o[1], o[2]);
    }
}

// CTA b: the tiles [b chunk, (b + 1) chunk) of the plane, row-major; each target block's
// sum over a run goes to the slot b - first(block).  R = 2: the mirror was written by
// na_stage_kernel; R = 1: every CTA converts what it reads (few CTAs read a particle while
// there are few target blocks, and a launch is saved).
template <int TENSOR, int R>
__global__ void __launch_bounds__(kThreads, kResident) na_dense_kernel(NaArgs a) {
    constexpr int TD = (TENSOR == T_OSEEN) ? T_OSEEN : T_RP;
    constexpr bool STAGED = R == 2;
    __shared__ __align__(16) float s_src[6 * kTile];
    const int tid = threadIdx.x, J = a.g.J;
    const size_t M = a.npad;
    const long long t0 = static_cast<long long>(blockIdx.x) * a.g.chunk, t1 = min(t0 + a.g.chunk, a.g.nT);
    f2 XI[R], YI[R], ZI[R];
    float hi[R][3], lo[R][3];
    int ib = static_cast<int>(t0 / a.g.nJT), jt = static_cast<int>(t0 - static_cast<long long>(ib) * a.g.nJT);
    bool fresh = true;
    for (long long t = t0; t < t1; ++t) {
        if (fresh) {
            fresh = false;
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const int i = ib * a.g.I + tid + k * kThreads;
                float v[6] = {-1.0e18f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};   // (not where padding sources are)
                if (STAGED) {
                    if (i < a.n)
                        for (int d = 0; d < 3; ++d) v[d] = a.mir[d * M + i];
                } else if (i < a.n) {
                    na_load(a, i, v);
                }
                XI[k] = pk2(v[0], v[0]);
                YI[k] = pk2(v[1], v[1]);
                ZI[k] = pk2(v[2], v[2]);
                for (int d = 0; d < 3; ++d) hi[k][d] = lo[k][d] = 0.0f;
            }
        }
        const int j0 = jt * J;
        if (STAGED) {
            for (int e = tid; e < 6 * J / 4; e += kThreads) {   // (J and npad: multiples of 4)
                const int d = e / (J / 4), q = e - d * (J / 4);
                reinterpret_cast<float4 *>(s_src)[e] = reinterpret_cast<const float4 *>(a.mir + d * M + j0)[q];
            }
        } else {
            for (int q = tid; q < J; q += kThreads) {
                float v[6];
                na_load(a, j0 + q, v);
                for (int d = 0; d < 6; ++d) s_src[d * J + q] = v[d];
            }
        }
        __syncthreads();
        f2 A[R][3];
#pragma unroll
        for (int k = 0; k < R; ++k) A[k][0] = A[k][1] = A[k][2] = 0ull;
        auto fold = [&]() {
#pragma unroll
            for (int k = 0; k < R; ++k)
                for (int d = 0; d < 3; ++d) {
                    float u, v;
                    upk2(A[k][d], u, v);
                    fold2(hi[k][d], lo[k][d], u);
                    fold2(hi[k][d], lo[k][d], v);
                    A[k][d] = 0ull;
                }
        };
        for (int jj = 0; jj < J; jj += 4) {
            if (jj == 128) fold();   // (at most 64 terms per packed lane between folds)
            f2 P[6][2];
#pragma unroll
            for (int d = 0; d < 6; ++d) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(s_src + d * J + jj);
                P[d][0] = v.x;
                P[d][1] = v.y;
            }
            f2 dx[R][2], dy[R][2], dz[R][2];
            float rr[R][4], mn = 3.0e38f;
#pragma unroll
            for (int k = 0; k < R; ++k)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    dx[k][h] = sub2(XI[k], P[0][h]);
                    dy[k][h] = sub2(YI[k], P[1][h]);
                    dz[k][h] = sub2(ZI[k], P[2][h]);
                    upk2(fma2(dz[k][h], dz[k][h], fma2(dy[k][h], dy[k][h], mul2(dx[k][h], dx[k][h]))), rr[k][2 * h],
                         rr[k][2 * h + 1]);
                    mn = fminf(mn, fminf(rr[k][2 * h], rr[k][2 * h + 1]));
                }
            if (mn < a.pc.r2min_f) {
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    float o[3] = {0.0f, 0.0f, 0.0f}, x, y, z, u;
                    upk2(XI[k], x, u);
                    upk2(YI[k], y, u);
                    upk2(ZI[k], z, u);
                    na_group<TENSOR>(x, y, z, s_src + jj, J, ib * a.g.I + tid + k * kThreads - j0 - jj, a.pc, o);
                    for (int d = 0; d < 3; ++d) A[k][d] = add2(A[k][d], pk2(o[d], 0.0f));
                }
                continue;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    const f2 ri = pk2(rsqrt_sfu(rr[k][2 * h]), rsqrt_sfu(rr[k][2 * h + 1])), ri2 = mul2(ri, ri);
                    f2 TA, TB;
                    if (TD == T_OSEEN) {
                        TA = mul2(a.c2.c1, ri);
                        TB = mul2(TA, ri2);
                    } else {
                        TA = mul2(ri, fma2(a.c2.c3, ri2, a.c2.c1));
                        TB = mul2(mul2(ri, ri2), fma2(a.c2.m3c3, ri2, a.c2.c1));
                    }
                    const f2 s = mul2(TB, fma2(dz[k][h], P[5][h], fma2(dy[k][h], P[4][h], mul2(dx[k][h], P[3][h]))));
                    A[k][0] = fma2(s, dx[k][h], fma2(TA, P[3][h], A[k][0]));
                    A[k][1] = fma2(s, dy[k][h], fma2(TA, P[4][h], A[k][1]));
                    A[k][2] = fma2(s, dz[k][h], fma2(TA, P[5][h], A[k][2]));
                }
        }
        fold();
        const bool row_end = ++jt == a.g.nJT;
        if (row_end || t + 1 == t1) {
            double *p = a.part + static_cast<size_t>(static_cast<int>(blockIdx.x) - geom_first(a.g, ib)) * 3 * M;
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const int i = ib * a.g.I + tid + k * kThreads;
                if (i < a.n)
                    for (int d = 0; d < 3; ++d) p[d * M + i] = static_cast<double>(hi[k][d]) + lo[k][d];
            }
        }
        if (row_end) {
            ++ib;
            jt = 0;
            fresh = true;
        }
        __syncthreads();   // the tile is free
    }
}

// V_i = mu0 (F_i + sum of the partials in slot order), FP64; one component per thread.
__global__ void na_finish_kernel(NaArgs a) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    const int d = q / a.npad, i = q - d * a.npad;   // (3 npad threads)
    if (i >= a.n) return;
    const int ib = i / a.g.I, ns = geom_last(a.g, ib) - geom_first(a.g, ib) + 1;
    const double *p = a.part + static_cast<size_t>(d) * a.npad + i;
    double v = a.F[3 * i + d];
#pragma unroll 4
    for (int s = 0; s < ns; ++s) v += p[static_cast<size_t>(s) * 3 * a.npad];
    a.V[3 * i + d] = a.pc.mu0 * v;
}

// From kPairN particles on, a thread takes two targets and the mirror is written by a kernel
// of its own; below, one target per thread spreads over more SMs and every CTA converts what
// it reads.  (Whole call, one side of the line: n = 4,095 48 us; the other: n = 4,096 54 us,
// 6,000 77 us against 62 us and 91 us before.)
constexpr int kPairN = 4096;

// The runs of tiles: tiles of 256 sources, or down to 64 while there are too few of them for
// every SM; up to eight equal waves of resident CTAs (the block scheduler evens out the SMs),
// as many as the scratch array has slots for.
DenseGeom na_geom(int n, int npad, int sms) {
    DenseGeom g{};
    const long long resident = static_cast<long long>(kResident) * sms;
    g.I = kThreads * (n >= kPairN ? 2 : 1);
    g.nIB = (n + g.I - 1) / g.I;
    for (g.J = kTile; ; g.J /= 2) {
        g.nJT = (n + g.J - 1) / g.J;
        g.nT = static_cast<long long>(g.nIB) * g.nJT;
        if (g.J == 64 || g.nT >= 4 * resident) break;
    }
    const long long slots = static_cast<long long>(kPartialDoubles) / (3LL * npad);   // >= kSplits
    for (int waves = 8; waves >= 1; --waves) {
        g.chunk = (g.nT + waves * resident - 1) / (waves * resident);
        if ((g.nJT + g.chunk - 1) / g.chunk + 1 <= slots) break;   // (a row meets at most that many runs)
    }
    while ((g.nJT + g.chunk - 1) / g.chunk + 1 > slots) ++g.chunk;
    g.grid = static_cast<int>((g.nT + g.chunk - 1) / g.chunk);
    return g;
}

template <int R>
void na_launch(int tensor, const NaArgs &g, cudaStream_t st) {
    switch (tensor) {
        case SD_TENSOR_RPY: na_dense_kernel<T_RPY, R><<<g.g.grid, kThreads, 0, st>>>(g); break;
        case SD_TENSOR_RP: na_dense_kernel<T_RP, R><<<g.g.grid, kThreads, 0, st>>>(g); break;
        default: na_dense_kernel<T_OSEEN, R><<<g.g.grid, kThreads, 0, st>>>(g); break;
    }
}

}  // namespace
}  // namespace sd

using namespace sd;

extern "C" sd_status sd_mobility_apply_noalloc(const double *x, const double *F, double *V, int32_t n, double a,
                                               double eta, int32_t tensor, void *stream) {
    if (n < 0) return set_error(SD_ERR_ARG, "n must be >= 0");
    if (n > kMaxN)
        return set_error(SD_ERR_ARG, "sd_mobility_apply_noalloc: n = " + std::to_string(n) +
                                         " exceeds the limit of its fixed scratch array (65536 particles)");
    if (!(a > 0.0) || !(eta > 0.0) || !std::isfinite(a) || !std::isfinite(eta))
        return set_error(SD_ERR_ARG, "a and eta must be finite and > 0");
    if (tensor < 0 || tensor > 2) return set_error(SD_ERR_ARG, "unknown tensor");
    if (n == 0) return SD_OK;
    if (!x || !F || !V) return set_error(SD_ERR_ARG, "x, F and V must be device pointers");
    void *base = nullptr;
    int sms = 0;
    sd_status s = noalloc_scratch(&base, &sms);
    if (s != SD_OK) return s;

    NaArgs g{};
    g.x = x;
    g.F = F;
    g.V = V;
    g.n = n;
    g.npad = ((n + kTile - 1) / kTile) * kTile;
    g.g = na_geom(n, g.npad, sms);
    g.mir = static_cast<float *>(base);
    g.part = reinterpret_cast<double *>(static_cast<unsigned char *>(base) + kMirrorFloats * sizeof(float));
    PairConst &pc = g.pc;
    pc.a = a;
    pc.two_a = 2.0 * a;
    pc.mu0 = 1.0 / (6.0 * 3.14159265358979323846 * eta * a);
    pc.r2min_d = 4.0 * a * a;
    pc.c1_d = 0.75 * a;
    pc.c3_d = 0.5 * a * a * a;
    pc.m3c3_d = -1.5 * a * a * a;
    pc.k_d = pc.c3_d / pc.c1_d;
    pc.m3k_d = -3.0 * pc.c3_d / pc.c1_d;
    pc.invc1_d = 1.0 / pc.c1_d;
    pc.r2min_f = static_cast<float>(pc.r2min_d);
    pc.c1_f = static_cast<float>(pc.c1_d);
    pc.c3_f = static_cast<float>(pc.c3_d);
    pc.m3c3_f = static_cast<float>(pc.m3c3_d);
    g.c2 = pair_const2(pc, n);

    // An error left by the caller's earlier work is reported as such and left in
    // place (peeked, not cleared); each launch below is then checked on its own.
    cudaError_t e = cudaPeekAtLastError();
    if (e != cudaSuccess)
        return set_error(SD_ERR_CUDA, std::string("sd_mobility_apply_noalloc: a CUDA error from earlier work is "
                                                  "pending (not cleared): ") + cudaGetErrorString(e));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool pair = n >= kPairN;
    if (pair) {
        na_stage_kernel<<<(g.npad + 127) / 128, 128, 0, st>>>(g);
        e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_status(e, "sd_mobility_apply_noalloc: staging launch");
    }
    if (pair) na_launch<2>(tensor, g, st);
    else na_launch<1>(tensor, g, st);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_status(e, "sd_mobility_apply_noalloc: all-pairs launch");
    na_finish_kernel<<<(3 * g.npad + 127) / 128, 128, 0, st>>>(g);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_status(e, "sd_mobility_apply_noalloc: reduction launch");
    return SD_OK;
}
