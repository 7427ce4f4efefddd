// Building blocks of the any-shape kernels (scans, layer norm, reductions, phase barrier, the FMA GEMM).
// Real = double in the fp64 kernels (fp32 I/O), float in the others.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "simt_layout.h"

namespace e2ttt {

constexpr int kSimtThreads = 256;
constexpr int kMaxC = 512;  // the paper trains with chunks of 512 tokens
constexpr int kMaxMat = 3;
constexpr int kBM = 64, kBN = 64, kBK = 16;
constexpr int kSM = 16, kSK = 64, kSplit = 4;  // the small tiling of the FMA GEMM

// ---- I/O conversion -------------------------------------------------------------------------
template <typename Real> __device__ __forceinline__ Real ld_io(const float* p, size_t i) { return (Real)p[i]; }
template <typename Real> __device__ __forceinline__ Real ld_io(const __nv_bfloat16* p, size_t i) {
    return (Real)__bfloat162float(p[i]);
}
template <typename Real> __device__ __forceinline__ void st_io(float* p, size_t i, Real v) { p[i] = (float)v; }
template <typename Real> __device__ __forceinline__ void st_io(__nv_bfloat16* p, size_t i, Real v) {
    p[i] = __float2bfloat16_rn((float)v);
}

// ---- scalar nonlinearities (exact erf GELU; Section 4 "Fast-weight Network") -------------------
__device__ __forceinline__ float r_erf(float x) { return erff(x); }
__device__ __forceinline__ double r_erf(double x) { return erf(x); }
__device__ __forceinline__ float r_exp(float x) { return expf(x); }
__device__ __forceinline__ double r_exp(double x) { return exp(x); }
__device__ __forceinline__ float r_rsqrt(float x) { return 1.0f / sqrtf(x); }
__device__ __forceinline__ double r_rsqrt(double x) { return 1.0 / sqrt(x); }

template <typename Real> __device__ __forceinline__ Real norm_cdf(Real z) {
    return (Real)0.5 * ((Real)1 + r_erf(z * (Real)0.70710678118654752440));
}
template <typename Real> __device__ __forceinline__ Real norm_pdf(Real z) {
    return (Real)0.39894228040143267794 * r_exp((Real)-0.5 * z * z);
}
template <typename Real> __device__ __forceinline__ Real gelu_f(Real z) { return z * norm_cdf(z); }
template <typename Real> __device__ __forceinline__ Real gelu_d1(Real z) { return norm_cdf(z) + z * norm_pdf(z); }
template <typename Real> __device__ __forceinline__ Real gelu_d2(Real z) { return norm_pdf(z) * ((Real)2 - z * z); }
template <typename Real> __device__ __forceinline__ Real sigmoid_f(Real z) { return (Real)1 / ((Real)1 + r_exp(-z)); }
template <typename Real> __device__ __forceinline__ Real silu_f(Real z) { return z * sigmoid_f(z); }
template <typename Real> __device__ __forceinline__ Real silu_d1(Real z) {
    Real s = sigmoid_f(z);
    return s * ((Real)1 + z * ((Real)1 - s));
}

// ---- warp helpers ------------------------------------------------------------------------------
__device__ __forceinline__ float shfl_down_r(float v, int off) { return __shfl_down_sync(0xffffffffu, v, off); }
__device__ __forceinline__ double shfl_down_r(double v, int off) { return __shfl_down_sync(0xffffffffu, v, off); }
__device__ __forceinline__ float shfl_xor_r(float v, int off) { return __shfl_xor_sync(0xffffffffu, v, off); }
__device__ __forceinline__ double shfl_xor_r(double v, int off) { return __shfl_xor_sync(0xffffffffu, v, off); }
template <typename Real> __device__ __forceinline__ Real warp_sum(Real v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += shfl_xor_r(v, off);
    return v;
}

// Deterministic CTA-wide sum (fixed tree); every thread gets the result. red: >= 16 Reals of shared memory.
template <typename Real> __device__ Real block_sum(Real v, Real* red) {
    v = warp_sum(v);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    Real s = 0;
    const int nw = (int)blockDim.x >> 5;
    for (int w = 0; w < nw; ++w) s += red[w];
    return s;
}

// ---- scalar kernels of a chunk -----------------------------------------------------------------
// Suffix scans over the gates of one chunk (Eq. "scalar_aux"), in the division-free form
//   gt_t = gamma_{t+1} gt_{t+1},  bt_t = beta_{t+1} bt_{t+1},  S_t = beta_{t+1} S_{t+1} + gt_t,   S_C = bt_C = gt_C = 1,
// where S_t = bt_t R_t is the weight of G_t in W_C (the inner sum of Eq. "unroll_recurrence").  A step is the
// linear map (bt, gt, S) -> (B bt, G gt, B S + X gt); maps compose associatively, so the suffix composites come
// from a warp-shuffle scan: each lane folds its own consecutive tokens, then five shuffle rounds fold the lanes.
template <typename Real> struct ScanMap { Real B, G, X; };
template <typename Real>
__device__ __forceinline__ ScanMap<Real> compose(const ScanMap<Real>& outer, const ScanMap<Real>& inner) {
    // inner acts first (it is nearer the chunk end), outer second
    ScanMap<Real> r;
    r.B = outer.B * inner.B;
    r.G = outer.G * inner.G;
    r.X = outer.B * inner.X + outer.X * inner.G;
    return r;
}

template <typename Real> struct ChunkScalars {
    Real kW[kMaxC];     // K^W_t = eta_t S_t          (token t at index t-1)
    Real kM[kMaxC];     // K^M_t = eta_t bt_t
    Real bt[kMaxC + 1]; // bt_t, t = 0..len
    Real gt[kMaxC + 1];
    Real S[kMaxC + 1];
    Real cw, cm, cb;    // gt_0, bt_0 R_1 = beta_1 S_1, bt_0
};

// Executed by one warp.  eta/beta/gamma point at the chunk's first token; len <= 32 EPL tokens, EPL per lane.  Out: ChunkScalars<Real> or
// a struct with the same names.
template <typename Real, int EPL, typename Out>
__device__ void chunk_scalars_scan(const float* eta, const float* beta, const float* gamma, int len, Out* out) {
    const int lane = threadIdx.x & 31;
    ScanMap<Real> local[EPL + 1];
    local[EPL].B = 1; local[EPL].G = 1; local[EPL].X = 0;
#pragma unroll
    for (int e = EPL - 1; e >= 0; --e) {
        const int i = lane * EPL + e;
        ScanMap<Real> m;
        if (i < len) { m.B = (Real)beta[i]; m.G = (Real)gamma[i]; m.X = m.G; }
        else { m.B = 1; m.G = 1; m.X = 0; }
        local[e] = compose(m, local[e + 1]);
    }
    ScanMap<Real> incl = local[0];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        ScanMap<Real> other;
        other.B = shfl_down_r(incl.B, off);
        other.G = shfl_down_r(incl.G, off);
        other.X = shfl_down_r(incl.X, off);
        if (lane + off < 32) incl = compose(incl, other);
    }
    ScanMap<Real> excl;
    excl.B = shfl_down_r(incl.B, 1);
    excl.G = shfl_down_r(incl.G, 1);
    excl.X = shfl_down_r(incl.X, 1);
    if (lane == 31) { excl.B = 1; excl.G = 1; excl.X = 0; }
#pragma unroll
    for (int e = 0; e <= EPL; ++e) {
        const int t = lane * EPL + e; // state index t = composite of tokens t+1..len
        if (e == EPL && lane != 31) continue; // same index as the next lane's e = 0
        if (t > len) continue;
        ScanMap<Real> f = compose(local[e], excl);
        out->bt[t] = f.B;
        out->gt[t] = f.G;
        out->S[t] = f.B + f.X;
    }
    __syncwarp();
    for (int i = lane; i < len; i += 32) {
        const Real e = (Real)eta[i];
        out->kW[i] = e * out->S[i + 1];
        out->kM[i] = e * out->bt[i + 1];
    }
    if (lane == 0) {
        out->cw = out->gt[0];
        out->cb = out->bt[0];
        out->cm = (Real)beta[0] * out->S[1];
    }
}
// A lane's own tokens are a serial chain in front of the shuffles, so short chunks take fewer per lane.
template <typename Real, typename Out>
__device__ void chunk_scalars_warp(const float* eta, const float* beta, const float* gamma, int len, Out* out) {
    if (len <= 64) chunk_scalars_scan<Real, 2>(eta, beta, gamma, len, out);
    else chunk_scalars_scan<Real, kMaxC / 32>(eta, beta, gamma, len, out);
}

// ---- launch of an any-shape kernel: N clusters of a.cl CTAs -------------------------------------
// `state`, per device: 0 nothing known, 1 the shared-memory limit is set, 8 or 16 the largest cluster the device grants
// `smem`: of this launch, `most`: of any launch of the kernel (what is asked of the device once holds for all); `more`: the kernel's further
// arguments
template <typename K, typename A, typename... Args>
int simt_launch(K kernel, A a, int threads, size_t smem, size_t most, std::atomic<int> (&state)[64], cudaStream_t st, Args... more) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return (int)e;
    const bool keep = dev >= 0 && dev < 64;
    int known = keep ? state[dev].load() : 0;
    if (known == 0) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
        if (e != cudaSuccess) return (int)e;
        known = 1;
    }
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = most;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    auto of = [&](int cl) {
        at[0].val.clusterDim.x = (unsigned)cl;
        cfg.gridDim = dim3((unsigned)(a.N * cl));
    };
    if (a.cl > 8) {
        if (known < 8)
            known = simt_granted_cluster(16, [&](int cl) {
                int n = 0;
                of(cl);
                if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
                    cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
                    (void)cudaGetLastError();
                    return 0;
                }
                return n;
            });
        if (a.cl > known) a.cl = known;
    }
    if (keep && known > state[dev].load()) state[dev] = known;
    of(a.cl);
    cfg.dynamicSmemBytes = smem;
    e = cudaLaunchKernelEx(&cfg, kernel, a, more...);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaGetLastError();
}

// ---- elementwise pass with batched loads ---------------------------------------------------------
// for e = begin, begin + stride, ... < end:  store(e, load(e)).  `load` returns everything element e needs from
// memory (a value or a small struct), `store` computes and writes.  U loads are issued before the U stores that
// follow them; written as one loop body, every load would wait for the previous element's store (the compiler must
// assume they alias) and the pass would take one memory round trip per element.
template <int U, typename FL, typename FS>
__device__ __forceinline__ void batched_for(size_t begin, size_t end, size_t stride, FL load, FS store) {
    using P = decltype(load((size_t)0));
    for (size_t e0 = begin; e0 < end; e0 += stride * U) {
        P p[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const size_t e = e0 + (size_t)u * stride;
            if (e < end) p[u] = load(e);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const size_t e = e0 + (size_t)u * stride;
            if (e < end) store(e, p[u]);
        }
    }
}

// ---- phase barrier ---------------------------------------------------------------------------------
// A sequence may be worked on by a cluster of `nranks` CTAs that split every phase (GEMM tiles, rows, elements)
// and share all intermediates through global memory.  The hardware cluster barrier (release / acquire at cluster
// scope) orders one phase's global writes before the next phase's reads; with one CTA it is the CTA barrier.
__device__ __forceinline__ void phase_sync(int nranks) {
    if (nranks == 1) {
        __syncthreads();
    } else {
        __syncwarp();  // .aligned: the warp's threads execute the instruction together, whatever branches came before
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// ---- generic CTA GEMM --------------------------------------------------------------------------
// out(m, n) = sum_k a(m, k) * b(n, k), m < M, n < N, k < K, for NACC (1 or 2) A operands sharing one B.
//   fa(m, k, a0, a1) writes the A value(s); fb(n, k) returns the B value; pre(m, n) loads what a result combines
//   with; epi(m, n, acc0, acc1, loaded) consumes a result.
// A_KFAST / B_KFAST say which index is contiguous in memory, so that neighbouring threads read neighbouring words.
// Two tilings, both ending with phase_sync(); the tiles are dealt round-robin to the `nranks` CTAs of the sequence's cluster:
//   64x64 tiles, 16-deep k slices, 4x4 results per thread: fewest loads per product, where there is a tile for every CTA;
//   16x16 tiles, 64-deep k slices cut four ways inside the CTA, 2x2 results per thread, the next slice's loads in flight while one
//   is multiplied: for the few tokens of a small problem.  A [32 x 64] result with 256 terms is one 64x64 tile - one CTA of
//   eight, half of its rows unused, 16 exposed round trips to L2 - but 8 small ones with 4 slices each.  Forward and reverse pass
//   (impl SIMT) of one sequence, large tiles alone -> both: 16 chunks of 16 tokens, d = 64, h = 256 5.53 -> 3.06 ms, 8 chunks of 64,
//   d = 128, h = 512 6.60 -> 6.49.
struct __align__(16) GemmSmem {
    union {
        struct {
            float A[2][kBK][kBM + 4];
            float B[kBK][kBN + 4];
        };
        struct {
            float2 a[2][kSK][kSM / 2 + 1];  // pairs: one access per two values
            float2 b[kSK][kSM / 2 + 1];
            float part[2][kSplit][kSM * kSM];
        } s;
    };
};

template <int NACC, bool A_KFAST, bool B_KFAST, typename FA, typename FB, typename FP, typename FE>
__device__ void block_gemm_small(int M, int N, int K, FA fa, FB fb, FP pre, FE epi, GemmSmem* sm, int rank, int nranks) {
    const int tid = threadIdx.x;
    const int grp = tid / (kSimtThreads / kSplit), tx = tid & 7, ty = (tid >> 3) & 7;
    const int tn = (N + kSM - 1) / kSM, tiles = tn * ((M + kSM - 1) / kSM);
    constexpr int PER = kSM * kSK / kSimtThreads;
    float ra0[PER], ra1[PER], rb[PER], acc[NACC][2][2];
    // the slice whose loads are in flight (the next one) and the slice in shared memory; divisions once per tile only
    int tile = rank, fm0 = (rank / tn) * kSM, fn0 = (rank % tn) * kSM, fk0 = 0;
    for (bool first = true;; first = false) {
        const int m0 = fm0, n0 = fn0, k0 = fk0;
        if (first) {
            if (tile >= tiles) break;
        } else {
            __syncthreads();
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                const int idx = tid + r * kSimtThreads;
                const int am = A_KFAST ? idx / kSK : idx % kSM, ak = A_KFAST ? idx % kSK : idx / kSM;
                const int bn = B_KFAST ? idx / kSK : idx % kSM, bk = B_KFAST ? idx % kSK : idx / kSM;
                const bool ina = m0 + am < M && k0 + ak < K, inb = n0 + bn < N && k0 + bk < K;
                reinterpret_cast<float*>(sm->s.a[0][ak])[am] = ina ? ra0[r] : 0.0f;
                if (NACC == 2) reinterpret_cast<float*>(sm->s.a[1][ak])[am] = ina ? ra1[r] : 0.0f;
                reinterpret_cast<float*>(sm->s.b[bk])[bn] = inb ? rb[r] : 0.0f;
            }
            __syncthreads();
            fk0 += kSK;
            if (fk0 >= K) {
                fk0 = 0;
                tile += nranks;
                fm0 = (tile / tn) * kSM;
                fn0 = (tile % tn) * kSM;
            }
        }
        if (tile < tiles) {
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                const int idx = tid + r * kSimtThreads;
                const int am = A_KFAST ? idx / kSK : idx % kSM, ak = A_KFAST ? idx % kSK : idx / kSM;
                const int bn = B_KFAST ? idx / kSK : idx % kSM, bk = B_KFAST ? idx % kSK : idx / kSM;
                // indices are clamped and the values masked when they are stored: no branch may stand between the loads, and
                // nothing may use a value before the multiplication that hides the loads
                ra0[r] = ra1[r] = 0;
                fa(min(fm0 + am, M - 1), min(fk0 + ak, K - 1), ra0[r], ra1[r]);
                rb[r] = fb(min(fn0 + bn, N - 1), min(fk0 + bk, K - 1));
            }
        }
        if (first) continue;
        const bool last_slice = k0 + kSK >= K;
        if (k0 == 0)
#pragma unroll
            for (int a = 0; a < NACC; ++a) acc[a][0][0] = acc[a][0][1] = acc[a][1][0] = acc[a][1][1] = 0;
        // what the tile's results combine with: on its way while the last slice is multiplied
        using P = decltype(pre(0, 0));
        P p;
        const int m = m0 + tid / kSM, n = n0 + tid % kSM;
        if (last_slice) p = pre(min(m, M - 1), min(n, N - 1));
        const int terms = min(kSK, K - k0);  // of this slice; dealt to the four groups in turn
#pragma unroll 4
        for (int kk = grp; kk < terms; kk += kSplit) {
            const float2 b = sm->s.b[kk][tx];
#pragma unroll
            for (int a = 0; a < NACC; ++a) {
                const float2 v = sm->s.a[a][kk][ty];
                acc[a][0][0] += v.x * b.x; acc[a][0][1] += v.x * b.y;
                acc[a][1][0] += v.y * b.x; acc[a][1][1] += v.y * b.y;
            }
        }
        if (last_slice) {
#pragma unroll
            for (int a = 0; a < NACC; ++a)
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 2; ++j) sm->s.part[a][grp][(2 * ty + i) * kSM + 2 * tx + j] = acc[a][i][j];
            __syncthreads();
            float s[2] = {0, 0};
#pragma unroll
            for (int a = 0; a < NACC; ++a)
#pragma unroll
                for (int g = 0; g < kSplit; ++g) s[a] += sm->s.part[a][g][tid];
            if (m < M && n < N) epi(m, n, s[0], s[NACC - 1], p);
            if (tile >= tiles) break;
        }
    }
}

template <int NACC, bool A_KFAST, bool B_KFAST, typename FA, typename FB, typename FP, typename FE>
__device__ void block_gemm(int M, int N, int K, FA fa, FB fb, FP pre, FE epi, GemmSmem* sm, int rank, int nranks) {
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    // fewer large tiles than CTAs, or a lone tile's row that is mostly padding: the small tiling keeps the cluster busy
    if (((M + kBM - 1) / kBM) * ((N + kBN - 1) / kBN) < nranks || 2 * M <= kBM || 2 * N <= kBN) {
        block_gemm_small<NACC, A_KFAST, B_KFAST>(M, N, K, fa, fb, pre, epi, sm, rank, nranks);
        phase_sync(nranks);
        return;
    }
    int tile = 0;
    for (int m0 = 0; m0 < M; m0 += kBM) {
        for (int n0 = 0; n0 < N; n0 += kBN, ++tile) {
            if (tile % nranks != rank) continue;
            float acc[NACC][4][4];
#pragma unroll
            for (int a = 0; a < NACC; ++a)
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[a][i][j] = 0;
            for (int k0 = 0; k0 < K; k0 += kBK) {
                __syncthreads();
#pragma unroll
                for (int r = 0; r < (kBM * kBK) / kSimtThreads; ++r) {
                    const int idx = tid + r * kSimtThreads;
                    const int mm = A_KFAST ? idx / kBK : idx % kBM;
                    const int kk = A_KFAST ? idx % kBK : idx / kBM;
                    float a0 = 0, a1 = 0;
                    if (m0 + mm < M && k0 + kk < K) fa(m0 + mm, k0 + kk, a0, a1);
                    sm->A[0][kk][mm] = a0;
                    if (NACC == 2) sm->A[1][kk][mm] = a1;
                }
#pragma unroll
                for (int r = 0; r < (kBN * kBK) / kSimtThreads; ++r) {
                    const int idx = tid + r * kSimtThreads;
                    const int nn = B_KFAST ? idx / kBK : idx % kBN;
                    const int kk = B_KFAST ? idx % kBK : idx / kBN;
                    float b = 0;
                    if (n0 + nn < N && k0 + kk < K) b = fb(n0 + nn, k0 + kk);
                    sm->B[kk][nn] = b;
                }
                __syncthreads();
#pragma unroll
                for (int kk = 0; kk < kBK; ++kk) {
                    float bv[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) bv[j] = sm->B[kk][tx * 4 + j];
#pragma unroll
                    for (int a = 0; a < NACC; ++a) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float av = sm->A[a][kk][ty * 4 + i];
#pragma unroll
                            for (int j = 0; j < 4; ++j) acc[a][i][j] += av * bv[j];
                        }
                    }
                }
            }
            // what the results combine with is loaded for the whole 4x4 block first (loads in flight together)
            using P = decltype(pre(0, 0));
            P p[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int m = m0 + ty * 4 + i, n = n0 + tx * 4 + j;
                    if (m < M && n < N) p[i][j] = pre(m, n);
                }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int m = m0 + ty * 4 + i, n = n0 + tx * 4 + j;
                    if (m < M && n < N) epi(m, n, acc[0][i][j], NACC == 2 ? acc[NACC - 1][i][j] : 0.0f, p[i][j]);
                }
        }
    }
    phase_sync(nranks);
}

// ---- layer norm of one row by one warp -----------------------------------------------------------
// Returns r = (var + eps)^(-1/2); writes y (may alias u).  d values, strided over the 32 lanes.
template <typename Real>
__device__ __forceinline__ Real warp_layernorm(const Real* u, Real* y, int d, Real eps) {
    const int lane = threadIdx.x & 31;
    Real s = 0;
    for (int i = lane; i < d; i += 32) s += u[i];
    const Real mu = warp_sum(s) / (Real)d;
    Real v = 0;
    for (int i = lane; i < d; i += 32) { const Real c = u[i] - mu; v += c * c; }
    const Real r = r_rsqrt(warp_sum(v) / (Real)d + eps);
    for (int i = lane; i < d; i += 32) y[i] = (u[i] - mu) * r;
    return r;
}

}  // namespace e2ttt
