// Engine of the block-tiled any-shape kernels: bulk copies of operand blocks -> shared memory ring -> tcgen05.mma ->
// tensor memory -> epilogue warps.  The kernels (tile_fwd.cu, tile_bwd.cu) are sequences of jobs; a job is one
// or more matrix products accumulated into up to two sets of tensor-memory columns, followed by an epilogue.
//
// 18 warps walk the same sequence of jobs in three roles: warp 16 copies operand blocks, warp 17 issues MMAs, warps 0-15
// run the epilogues (warp w owns tensor-memory lanes 32 (w & 3).. and a quarter of the columns, w >> 2).
//
// Arithmetic: every fp32 operand x is two bf16 numbers, hi = bf16(x) and lo = bf16(x - hi), and a product is three MMAs,
// hi hi + hi lo + lo hi (the dropped lo lo term and the residual of the split are ~2^-16 relative), fp32 accumulation.
// The tokens are bf16 to begin with and have no lo part: two MMAs.
//
// All products put a feature dimension (d or hidden units) on the 128 tensor-memory lanes and tokens (or the other feature
// dimension) on the columns, so the epilogues' global accesses run along the contiguous index of every fp32 array.
// A block is stored once and read both ways: contraction along its rows' 64 columns (K-major) or down its 64 rows
// (MN-major), see sm100.cuh.
#pragma once
#include "simt_common.cuh"
#include "sm100.cuh"
#include "tile_layout.h"

namespace e2ttt {
namespace tile {

using namespace sm100;

constexpr int kEpiWarps = 16;
constexpr int kThreads = (kEpiWarps + 2) * 32;
constexpr int kEpiThreads = kEpiWarps * 32;
constexpr int kUnits = 6;             // ring: operand slices of 128 x 64 (hi rows 0-127, lo rows 0-127)
constexpr uint32_t kUnitBytes = 32768;
constexpr uint32_t kHalf = 8192;      // one 64 x 64 bf16 block
constexpr uint32_t kAccCols = 256;    // tensor-memory columns of one accumulator set; two sets

struct Sync {
    uint64_t full[kUnits], empty[kUnits], acc_full[2], acc_empty[2];
    uint32_t tmem;
    int dead;
};

// One 128 x 64 operand: two blocks (or one: 64 x 64), advancing by `ks` bytes per 64 k.
struct Opnd {
    const unsigned char* p0;
    const unsigned char* p1;  // second block along M / N; nullptr: none
    uint32_t ks;
    bool lo;                  // has a lo part (behind the hi part)
    bool mn;                  // the 64 columns of a block run along M / N, its rows along k
};

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
// bytes and address multiples of 16
__device__ __forceinline__ void l2_prefetch(const void* p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }

struct Engine {
    uint32_t ring;  // shared-memory address of the ring (1024-byte aligned)
    Sync* sy;
    uint32_t tmem;
    WaitCtx wc;
    int warp, lane;
    int rank, nranks;
    uint32_t unit = 0;  // operand slices loaded / consumed so far
    uint32_t job = 0;   // jobs so far; job & 1 = accumulator set
    uint32_t started = 0;  // MMA warp: accumulators of the current job that hold something

    __device__ bool epi() const { return warp < kEpiWarps; }

    __device__ void setup(unsigned char* ring_ptr, Sync* s, int* status, int rank_, int nranks_) {
        ring = smem_u32(ring_ptr);
        sy = s;
        // From lane 0: the compiler then knows that it is the same for the warp, and keeps what follows from it - the MMAs' descriptors - in
        // uniform registers
        warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
        lane = threadIdx.x & 31;
        rank = rank_;
        nranks = nranks_;
        if (threadIdx.x == 0) {
            for (int i = 0; i < kUnits; ++i) { mbar_init(&s->full[i], 1); mbar_init(&s->empty[i], 1); }
            for (int i = 0; i < 2; ++i) { mbar_init(&s->acc_full[i], 1); mbar_init(&s->acc_empty[i], kEpiWarps); }
            s->dead = 0;
            fence_mbar_init();
        }
        if (warp == 0) {
            tmem_alloc(&s->tmem, 512);
            tmem_relinquish();
        }
        tc_fence_before_sync();
        __syncthreads();
        tc_fence_after_sync();
        tmem = __shfl_sync(0xffffffffu, s->tmem, 0);
        wc.dead = &s->dead;
        wc.status = status;
    }
    __device__ void teardown() {
        tc_fence_before_sync();
        __syncthreads();
        if (*wc.dead) {  // a wait has given up: copies nobody waited for may still be under way to this CTA's shared memory
            const long long t0 = clock64();
            while (clock64() - t0 < 8000000) {}
            __syncthreads();
        }
        if (warp == 0) tmem_dealloc(tmem, 512);
    }

    // Phase barriers.  Operand blocks are written with plain stores and read by bulk copies (another proxy): fenced on
    // both sides.
    __device__ void sync_cta() {
        fence_proxy_async_all();
        __syncthreads();
        fence_proxy_async_all();
    }
    __device__ void sync_cluster() {
        fence_proxy_async_all();
        __syncwarp();
        phase_sync(nranks);
        fence_proxy_async_all();
    }

    __device__ void load(const Opnd& o, int k) {  // copy warp
        const uint32_t u = unit % kUnits, use = unit / kUnits;
        ++unit;
        if (use > 0) mbar_wait(&sy->empty[u], (use - 1) & 1, wc, 301);
        if (lane == 0) {
            const uint32_t dst = ring + u * kUnitBytes;
            const size_t off = (size_t)k * o.ks;
            const int n = o.p1 ? 2 : 1;
            mbar_expect_tx(&sy->full[u], (uint32_t)n * kHalf * (o.lo ? 2u : 1u));
            bulk_g2s(dst, o.p0 + off, kHalf, &sy->full[u]);
            if (o.p1) bulk_g2s(dst + kHalf, o.p1 + off, kHalf, &sy->full[u]);
            if (o.lo) {
                bulk_g2s(dst + 2 * kHalf, o.p0 + off + kHalf, kHalf, &sy->full[u]);
                if (o.p1) bulk_g2s(dst + 3 * kHalf, o.p1 + off + kHalf, kHalf, &sy->full[u]);
            }
        }
        __syncwarp();
    }

    __device__ void job_begin() {
        if (warp == kEpiWarps + 1) {
            if (job >= 2) mbar_wait(&sy->acc_empty[job & 1], ((job >> 1) - 1) & 1, wc, 302);
            tc_fence_after_sync();
            started = 0;
        }
    }

    // sum over nk slices of 64 k:  D[col[i]] += S P[i]^T  for i < np, with S on the lane side (s_lane) or the column side.
    // `col`: first column of the accumulator inside the job's set.  SPLIT: the products with a lo part in the 128 columns behind it, for
    // contractions of many slices (every MMA onto the sum truncates it; theirs are 2^-9 of it), added by the epilogue.
    template <int NP, bool SPLIT = false> __device__ void term(int nk, bool s_lane, const Opnd& s, const Opnd (&p)[NP], const uint32_t (&col)[NP]) {
        if (warp == kEpiWarps) {
            for (int k = 0; k < nk; ++k) {
                load(s, k);
#pragma unroll
                for (int i = 0; i < NP; ++i) load(p[i], k);
            }
        } else if (warp == kEpiWarps + 1) {
            const bool issue = lane == 0;
            for (int k = 0; k < nk; ++k) {
                const uint32_t us = unit % kUnits;
                mbar_wait(&sy->full[us], (unit / kUnits) & 1, wc, 303);
                ++unit;
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    const uint32_t up = unit % kUnits;
                    mbar_wait(&sy->full[up], (unit / kUnits) & 1, wc, 304);
                    ++unit;
                    tc_fence_after_sync();
                    const Opnd& a = s_lane ? s : p[i];
                    const Opnd& b = s_lane ? p[i] : s;
                    const uint32_t ua = ring + (s_lane ? us : up) * kUnitBytes, ub = ring + (s_lane ? up : us) * kUnitBytes;
                    const uint32_t idesc = make_idesc(128, b.p1 ? 128 : 64, a.mn, b.mn);
                    const uint32_t sa = a.mn ? 2048u : 32u, sb = b.mn ? 2048u : 32u;
                    const uint32_t d = tmem + (job & 1) * kAccCols + col[i];
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) {
                        const uint64_t ah = make_smem_desc(ua + ks * sa, kHalf, 1024), bh = make_smem_desc(ub + ks * sb, kHalf, 1024);
                        const uint64_t al = ah + (2 * kHalf >> 4), bl = bh + (2 * kHalf >> 4);
                        bool acc = (started >> i & 1u) || ks > 0;
                        if constexpr (SPLIT) {
                            bool acl = acc;
                            if (a.lo) { umma_bf16_elect(d + 128, al, bh, idesc, acl, issue); acl = true; }
                            if (b.lo) umma_bf16_elect(d + 128, ah, bl, idesc, acl, issue);
                        } else {
                            if (a.lo) { umma_bf16_elect(d, al, bh, idesc, acc, issue); acc = true; }  // small terms first
                            if (b.lo) { umma_bf16_elect(d, ah, bl, idesc, acc, issue); acc = true; }
                        }
                        umma_bf16_elect(d, ah, bh, idesc, acc, issue);
                    }
                    started |= 1u << i;
                    umma_commit_elect(&sy->empty[up], issue);
                }
                umma_commit_elect(&sy->empty[us], issue);
            }
        }
    }

    // f(t): epilogue of one warp; t = tensor-memory address of the set at this warp's lanes
    template <typename F> __device__ void job_end(F f) {
        if (warp == kEpiWarps + 1) {
            umma_commit_elect(&sy->acc_full[job & 1], lane == 0);
        } else if (warp < kEpiWarps) {
            mbar_wait(&sy->acc_full[job & 1], (job >> 1) & 1, wc, 305);
            tc_fence_after_sync();
            f(tmem + (job & 1) * kAccCols + ((uint32_t)(32 * (warp & 3)) << 16));
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sy->acc_empty[job & 1]);
        }
        ++job;
    }
};

// ---- operand blocks -----------------------------------------------------------------------------------------------------
// 16 consecutive values of one block row (col0 a multiple of 16), as one 32-byte store per part: hi at blk, lo at blk + 8192
__device__ __forceinline__ void st_split16(unsigned char* blk, int row, int col0, const float (&v)[16]) {
    uint32_t h[8], l[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const __nv_bfloat162 hh = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
        const float2 hf = __bfloat1622float2(hh);
        h[j] = *reinterpret_cast<const uint32_t*>(&hh);
        l[j] = pack_bf16(v[2 * j] - hf.x, v[2 * j + 1] - hf.y);
    }
    // pieces c and c + 1 (c even) share a 32-byte sector after the swizzle, in swapped order on odd rows
    const bool sw = row & 1;
    unsigned char* p = blk + row * 128 + ((((col0 >> 3) ^ (row & 7)) & ~1) << 4);
#pragma unroll
    for (int part = 0; part < 2; ++part) {
        const uint32_t* w = part ? l : h;
        asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p + part * kHalf), "r"(sw ? w[4] : w[0]),
                     "r"(sw ? w[5] : w[1]), "r"(sw ? w[6] : w[2]), "r"(sw ? w[7] : w[3]), "r"(sw ? w[0] : w[4]), "r"(sw ? w[1] : w[5]),
                     "r"(sw ? w[2] : w[6]), "r"(sw ? w[3] : w[7])
                     : "memory");
    }
}
// 16 consecutive values of one row of a 64 x 64 block in shared memory (hi; lo `lo` bytes behind)
__device__ __forceinline__ void sts_split16(uint32_t blk, uint32_t lo, int row, int col0, const float (&v)[16]) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        uint32_t h[4], l[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float x = v[8 * c + 2 * j], y = v[8 * c + 2 * j + 1];
            const __nv_bfloat162 hh = __floats2bfloat162_rn(x, y);
            const float2 hf = __bfloat1622float2(hh);
            h[j] = *reinterpret_cast<const uint32_t*>(&hh);
            l[j] = pack_bf16(x - hf.x, y - hf.y);
        }
        const uint32_t at = blk + row * 128 + ((((col0 >> 3) + c) ^ (row & 7)) << 4);
        asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(at), "r"(h[0]), "r"(h[1]), "r"(h[2]), "r"(h[3]) : "memory");
        asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(at + lo), "r"(l[0]), "r"(l[1]), "r"(l[2]), "r"(l[3]) : "memory");
    }
}
// 8 consecutive floats, 32-byte aligned
__device__ __forceinline__ void st_f8(float* p, const float (&v)[8]) {
    asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}
__device__ __forceinline__ void ld_f8(const float* p, float (&v)[8]) {
    asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p)
                 : "memory");
}
// hi + lo of 16 consecutive values
__device__ __forceinline__ void ld_split16(const unsigned char* blk, int row, int col0, float (&v)[16]) {
    const bool sw = row & 1;
    const unsigned char* p = blk + row * 128 + ((((col0 >> 3) ^ (row & 7)) & ~1) << 4);
    uint32_t w[2][8];
#pragma unroll
    for (int part = 0; part < 2; ++part)
        asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(w[part][0]), "=r"(w[part][1]), "=r"(w[part][2]), "=r"(w[part][3]), "=r"(w[part][4]), "=r"(w[part][5]),
                       "=r"(w[part][6]), "=r"(w[part][7])
                     : "l"(p + part * kHalf)
                     : "memory");
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint32_t hw = sw ? w[0][(j + 4) & 7] : w[0][j], lw = sw ? w[1][(j + 4) & 7] : w[1][j];
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&hw));
        const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&lw));
        v[2 * j] = a.x + b.x;
        v[2 * j + 1] = a.y + b.y;
    }
}
// 4 consecutive values of a block row (col a multiple of 4); LO = false: hi only
template <bool LO> __device__ __forceinline__ void st_split4(unsigned char* blk, int row, int col, const float (&v)[4]) {
    const __nv_bfloat162 h0 = __floats2bfloat162_rn(v[0], v[1]), h1 = __floats2bfloat162_rn(v[2], v[3]);
    unsigned char* p = blk + row * 128 + (((col >> 3) ^ (row & 7)) << 4) + ((col & 4) << 1);
    *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
    if (LO) {
        const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
        *reinterpret_cast<uint2*>(p + kHalf) = make_uint2(pack_bf16(v[0] - f0.x, v[1] - f0.y), pack_bf16(v[2] - f1.x, v[3] - f1.y));
    }
}

__device__ __forceinline__ void acc8(uint32_t t, float (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(t)
                 : "memory");
    tmem_wait_ld();
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[j]);
}
__device__ __forceinline__ void acc16(uint32_t t, float (&v)[16]) {
    uint32_t r[16];
    tmem_ld16(t, r);
    tmem_wait_ld();
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// Sums of 16 values over the 32 lanes: lane l returns the sum of v[l >> 1].  16 shuffles.
__device__ __forceinline__ float reduce16(const float (&v)[16], int lane) {
    float a[8], b[4], c[2];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float keep = (lane & 16) ? v[j + 8] : v[j], give = (lane & 16) ? v[j] : v[j + 8];
        a[j] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float keep = (lane & 8) ? a[j + 4] : a[j], give = (lane & 8) ? a[j] : a[j + 4];
        b[j] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const float keep = (lane & 4) ? b[j + 2] : b[j], give = (lane & 4) ? b[j] : b[j + 2];
        c[j] = keep + __shfl_xor_sync(0xffffffffu, give, 4);
    }
    const float keep = (lane & 2) ? c[1] : c[0], give = (lane & 2) ? c[0] : c[1];
    const float s = keep + __shfl_xor_sync(0xffffffffu, give, 2);
    return s + __shfl_xor_sync(0xffffffffu, s, 1);
}

// ---- activations ---------------------------------------------------------------------------------------------------------------
// The epilogues evaluate them for every token and hidden unit, and were bound by the instructions of erff, expf and the division.
// Normal distribution function and density: erfc(x) = t exp(P(t) - x^2), t = 1 / (1 + x / 2), the form of Press et al., Numerical Recipes
// (erfc by Chebyshev fitting), with a fit of its own: P of degree 9 to log(exp(x^2) erfc(x) / t) on t in [0.15, 1], error 6e-8 (beyond,
// at |z| > 16, the tail is 0 in fp32).  The distribution function is within 2.6e-7 in fp32, to which the hardware's exponential (3 ulp)
// and division (2 ulp) may add 3e-7; the products that follow round to 16 bits of mantissa.  The reverse pass recomputes the activations with erff (tile_rec.cuh); the two are as far apart.
__device__ __forceinline__ void normal_dist(float z, float& cdf, float& pdf) {
    const float x = 0.70710678118f * fabsf(z), x2 = x * x;
    const float t = __fdividef(1.0f, fmaf(0.5f, x, 1.0f));
    float p = fmaf(t, 0.154191726f, -0.731059300f);
    p = fmaf(t, p, 1.274361592f);
    p = fmaf(t, p, -0.851879440f);
    p = fmaf(t, p, 0.047508604f);
    p = fmaf(t, p, -0.066028275f);
    p = fmaf(t, p, 0.057246348f);
    p = fmaf(t, p, 0.381963899f);
    p = fmaf(t, p, 0.999168800f);
    p = fmaf(t, p, -1.265473900f);
    const float q = 0.5f * t * __expf(p - x2);  // P(Z > |z|)
    cdf = z < 0.0f ? q : 1.0f - q;
    pdf = 0.39894228040f * __expf(-x2);
}
__device__ __forceinline__ float sigmoid_hw(float z) { return __fdividef(1.0f, 1.0f + __expf(-z)); }

// ---- rows of the caller's bf16 token tensors: 4 values at column c (0 beyond d) -----------------------------------------
__device__ __forceinline__ void ld_tok4(const __nv_bfloat16* row, int c, int d, float (&v)[4]) {
    if ((d & 3) == 0) {
        uint2 raw = make_uint2(0u, 0u);
        if (c < d) raw = *reinterpret_cast<const uint2*>(row + c);
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.x));
        const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.y));
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = c + j < d ? __bfloat162float(row[c + j]) : 0.0f;
    }
}
__device__ __forceinline__ void st_tok4(__nv_bfloat16* row, int c, int d, const float (&v)[4]) {
    if ((d & 3) == 0) {
        if (c < d) *reinterpret_cast<uint2*>(row + c) = make_uint2(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]));
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (c + j < d) row[c + j] = __float2bfloat16_rn(v[j]);
    }
}
// v += p[0] + p[stride] + .., in that order, U loads in flight
template <int U = 4> __device__ __forceinline__ void add_parts(const float* p, int n, size_t stride, float (&v)[4]) {
    for (int i0 = 0; i0 < n; i0 += U) {
        float4 x[U];
#pragma unroll
        for (int i = 0; i < U; ++i)
            x[i] = i0 + i < n ? *reinterpret_cast<const float4*>(p + (size_t)(i0 + i) * stride) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < U; ++i) { v[0] += x[i].x; v[1] += x[i].y; v[2] += x[i].z; v[3] += x[i].w; }
    }
}
// warp-wide sums of R values, R independent shuffles in flight
template <int R> __device__ __forceinline__ void warp_sums(float (&v)[R]) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        float o[R];
#pragma unroll
        for (int i = 0; i < R; ++i) o[i] = __shfl_xor_sync(0xffffffffu, v[i], off);
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] += o[i];
    }
}
__device__ __forceinline__ float sum4(const float (&a)[4]) { return (a[0] + a[1]) + (a[2] + a[3]); }
__device__ __forceinline__ float dot4(const float (&a)[4], const float (&b)[4]) {
    return (a[0] * b[0] + a[1] * b[1]) + (a[2] * b[2] + a[3] * b[3]);
}

// Tokens of one chunk -> blocks (rows = tokens, hi only; rows past `len` and columns past d are zero).  `first` / `step`
// pick the rows of the calling warp out of tb * 64.
__device__ __forceinline__ void tokens_to_blocks(const __nv_bfloat16* src, int len, int d, int db, int tb, unsigned char* dst, int first, int step,
                                                 int lane) {
    constexpr int R = 4;  // rows in flight
    for (int t0 = first; t0 < tb * 64; t0 += R * step) {
        float v[R][4];
#pragma unroll
        for (int i = 0; i < R; ++i) ld_tok4(src + (size_t)min(t0 + i * step, len - 1) * d, 4 * lane, d, v[i]);
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int t = t0 + i * step;
            if (t >= len)
#pragma unroll
                for (int j = 0; j < 4; ++j) v[i][j] = 0.0f;
            if (t < tb * 64 && 4 * lane < db * 64) st_split4<false>(dst + (size_t)((t >> 6) * db + (lane >> 4)) * kHalf, t & 63, (4 * lane) & 63, v[i]);
        }
    }
}

// A row-major fp32 matrix [slow][fast] -> blocks whose rows are the FAST index and whose columns are the slow one, for the
// 64-blocks [fb0, fb1) x [sb0, sb1).  The calling warps (`w` of `nw`) deal the (32 fast x 16 slow) pieces among themselves.
// Block (fast / 64, slow / 64) sits at ((fast / 64) * rs + (slow / 64) * cs) * 16 KB.
__device__ __forceinline__ void matrix_to_blocks(const float* src, int nfast, int nslow, int fb0, int fb1, int sb0, int sb1, unsigned char* dst, int rs,
                                                 int cs, int w, int nw, int lane) {
    const int nf = (fb1 - fb0) * 2, pieces = nf * (sb1 - sb0) * 4;
    for (int e = w; e < pieces; e += nw) {
        const int f = fb0 * 64 + 32 * (e % nf) + lane, s0 = sb0 * 64 + 16 * (e / nf);
        float v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = src[(size_t)min(s0 + j, nslow - 1) * nfast + min(f, nfast - 1)];
        if (f >= nfast || s0 + 16 > nslow)
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = (f < nfast && s0 + j < nslow) ? v[j] : 0.0f;
        st_split16(dst + ((size_t)(f >> 6) * rs + (size_t)(s0 >> 6) * cs) * (2 * kHalf), f & 63, s0 & 63, v);
    }
}

}  // namespace tile
}  // namespace e2ttt
