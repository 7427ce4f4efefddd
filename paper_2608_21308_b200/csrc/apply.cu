// Outputs of fixed fast weights: o_t = f_W(q_t) = q_t + LN(W_last act(W_first q_t)) for T tokens per sequence, no update.
// This is the decode path between chunk boundaries (Algorithm 1 line 1 with the chunk-start weights; the state only
// changes once a whole chunk of keys and values has accumulated, and that step is e2ttt_chunk_fwd on those tokens).
//
// For a handful of tokens the work is a matrix-vector product over the whole state, so the kernel is bound by reading
// W once from HBM: 4 * nmat * d * h bytes per sequence.  A cluster of up to 8 CTAs serves one sequence; CTA c streams
// the hidden units [h0, h1) of every matrix - rows of the first matrices, a column slice of the last - with 8
// independent 16-byte loads per lane in flight, keeps the activations of its slice in shared memory, and produces a
// partial sum of the d outputs.  The slice of the last matrix does not depend on the activations, so its copy into
// shared memory (cp.async, no registers) is started before the first matrices are read: all of a CTA's bytes are in
// flight together.  The partial sums meet in the shared memory of the cluster's first CTA (distributed
// shared memory, fixed summation order), which applies the layer norm and the residual and stores o.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>

#include "apply.h"
#include "simt_common.cuh"
#include "sm100.cuh"

namespace cg = cooperative_groups;

namespace e2ttt {
namespace {

constexpr int kApThreads = 256;
constexpr int kApWarps = kApThreads / 32;
constexpr int kApHB = 256;   // hidden units per pass through shared memory
constexpr int kApRows = 8;   // rows a warp streams at once (independent loads in flight)
constexpr int kApStageBytes = 64 * 1024;  // shared-memory staging of the last matrix's block (asynchronous copies)

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)), "l"(gmem_src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}

template <typename T> __device__ __forceinline__ float ap_ld(const T* p, size_t i);
template <> __device__ __forceinline__ float ap_ld<float>(const float* p, size_t i) { return p[i]; }
template <> __device__ __forceinline__ float ap_ld<__nv_bfloat16>(const __nv_bfloat16* p, size_t i) { return __bfloat162float(p[i]); }
__device__ __forceinline__ void ap_st(float* p, size_t i, float v) { p[i] = v; }
__device__ __forceinline__ void ap_st(__nv_bfloat16* p, size_t i, float v) { p[i] = __float2bfloat16(v); }

// dot products of R rows of a row-major matrix (row stride ld, columns [c0, c0 + n)) with TB vectors held in shared
// memory (x[t][0..n)); one warp, result valid in every lane.  VEC: 16-byte loads (n % 4 == 0, aligned rows).
template <int R, int TB, bool VEC>
__device__ __forceinline__ void warp_dots(const float* __restrict__ w, size_t ld, int rows_valid, int n,
                                          const float* x, int xld, float (&acc)[R][TB]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int t = 0; t < TB; ++t) acc[r][t] = 0.0f;
    if (VEC) {
        for (int c = 4 * lane; c < n; c += 128) {
            float4 wv[R];
#pragma unroll
            for (int r = 0; r < R; ++r)
                wv[r] = (r < rows_valid) ? *reinterpret_cast<const float4*>(w + (size_t)r * ld + c) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int t = 0; t < TB; ++t) {
                const float4 xv = *reinterpret_cast<const float4*>(x + (size_t)t * xld + c);
#pragma unroll
                for (int r = 0; r < R; ++r)
                    acc[r][t] += wv[r].x * xv.x + wv[r].y * xv.y + wv[r].z * xv.z + wv[r].w * xv.w;
            }
        }
    } else {
        for (int c = lane; c < n; c += 32) {
            float wv[R];
#pragma unroll
            for (int r = 0; r < R; ++r) wv[r] = (r < rows_valid) ? w[(size_t)r * ld + c] : 0.0f;
#pragma unroll
            for (int t = 0; t < TB; ++t) {
                const float xv = x[(size_t)t * xld + c];
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r][t] += wv[r] * xv;
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int t = 0; t < TB; ++t) acc[r][t] = warp_sum(acc[r][t]);
}

template <typename IO, int KIND, int TB, bool VEC>
__global__ void __launch_bounds__(kApThreads, 2) apply_kernel(const ApplyArgs a) {
    constexpr int NMAT = (KIND == 0) ? 2 : 3;
    extern __shared__ __align__(16) float ap_smem[];
    cg::cluster_group cluster = cg::this_cluster();
    const int CL = a.cl;
    const int seq = blockIdx.x / CL, rank = blockIdx.x % CL;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int d = a.d, h = a.h, T = a.T;
    const size_t dh = (size_t)d * h;

    float* qs = ap_smem;                       // [TB][d]   the tokens
    float* as = qs + (size_t)TB * d;           // [TB][HB]  activations of the current hidden block
    float* up = as + (size_t)TB * kApHB;       // [TB][d]   this CTA's partial sums
    float* slots = up + (size_t)TB * d;        // [CL][TB][d] on the first CTA: every CTA's partial sums
    float* wls = slots + (size_t)CL * TB * d;  // [d][nh] staged block of the last matrix (when a.stage)

    const IO* q = reinterpret_cast<const IO*>(a.q) + (size_t)seq * T * d;
    IO* o = reinterpret_cast<IO*>(a.o) + (size_t)seq * T * d;
    const float* W1 = a.W[0] + (size_t)seq * dh;                                 // [h, d]
    const float* W2 = (KIND == 1) ? a.W[1] + (size_t)seq * dh : nullptr;         // [h, d] (SwiGLU gate partner)
    const float* Wl = a.W[NMAT - 1] + (size_t)seq * dh;                          // [d, h]

    // this CTA's hidden units: an even split in multiples of 4 (keeps 16-byte alignment of the column slices)
    const int per = ((h + CL - 1) / CL + 3) & ~3;
    const int h0 = min(h, rank * per), h1 = min(h, h0 + per);
    float* slot0 = cluster.map_shared_rank(slots, 0);

    // Programmatic dependent launch: this grid may start while the previous kernel of the stream is still running.
    // Nothing it produces may be touched before griddepcontrol.wait - but the fast weights of this CTA can already be
    // pulled from HBM into L2 (a prefetch has no effect on memory contents), so that the next layer's weights stream
    // in under the tail of the previous kernel.  Without a programmatic predecessor the wait returns at once.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (h0 < h1) {
        const int nrows = h1 - h0;
        // rows [h0, h1) of the first matrices are contiguous; the last matrix contributes d row segments
        const size_t bytes1 = (size_t)nrows * d * sizeof(float);
        for (size_t off = (size_t)tid * 128; off < bytes1; off += (size_t)kApThreads * 128) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(W1 + (size_t)h0 * d) + off));
            if (KIND == 1) asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(W2 + (size_t)h0 * d) + off));
        }
        const int seg = (nrows * (int)sizeof(float) + 127) / 128;  // 128-byte lines per row segment
        for (int e = tid; e < d * seg; e += kApThreads) {
            const int i = e / seg, c = e - i * seg;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(Wl + (size_t)i * h + h0) + (size_t)c * 128));
        }
    }
    // shared memory of another CTA may be touched only once that CTA runs: arrived here, waited for before the first store there
    sm100::cluster_arrive();
    asm volatile("griddepcontrol.wait;" ::: "memory");

    for (int t0 = 0; t0 < T; t0 += TB) {
        const int tb = min(TB, T - t0);
        for (int e = tid; e < TB * d; e += kApThreads) {
            const int t = e / d, i = e - t * d;
            qs[e] = (t < tb) ? ap_ld<IO>(q, (size_t)(t0 + t) * d + i) : 0.0f;
            up[e] = 0.0f;
        }
        __syncthreads();
        for (int hb = h0; hb < h1; hb += kApHB) {
            const int nh = min(kApHB, h1 - hb);
            if (VEC && a.stage) {  // start the copy of the last matrix's block; it lands while the activations are computed
                const int n4 = nh >> 2;
                for (int e = tid; e < d * n4; e += kApThreads) {
                    const int i = e / n4, c4 = e - i * n4;
                    cp_async16(wls + (size_t)i * nh + 4 * c4, Wl + (size_t)i * h + hb + 4 * c4);
                }
            }
            // hidden activations of the block: one warp per group of rows
            for (int j0 = warp * kApRows; j0 < nh; j0 += kApWarps * kApRows) {
                const int rv = min(kApRows, nh - j0);
                float z1[kApRows][TB];
                warp_dots<kApRows, TB, VEC>(W1 + (size_t)(hb + j0) * d, d, rv, d, qs, d, z1);
                if (KIND == 1) {
                    float z2[kApRows][TB];
                    warp_dots<kApRows, TB, VEC>(W2 + (size_t)(hb + j0) * d, d, rv, d, qs, d, z2);
#pragma unroll
                    for (int r = 0; r < kApRows; ++r)
#pragma unroll
                        for (int t = 0; t < TB; ++t) z1[r][t] = silu_f(z1[r][t]) * z2[r][t];
                } else {
#pragma unroll
                    for (int r = 0; r < kApRows; ++r)
#pragma unroll
                        for (int t = 0; t < TB; ++t) z1[r][t] = gelu_f(z1[r][t]);
                }
                if (lane == 0) {
#pragma unroll
                    for (int r = 0; r < kApRows; ++r)
                        if (r < rv)
#pragma unroll
                            for (int t = 0; t < TB; ++t) as[(size_t)t * kApHB + j0 + r] = z1[r][t];
                }
            }
            // zero the tail so that the vector loop below may run over a multiple of 4
            for (int e = tid; e < TB * 4; e += kApThreads) {
                const int t = e >> 2, j = nh + (e & 3);
                if (j < kApHB) as[(size_t)t * kApHB + j] = 0.0f;
            }
            if (VEC && a.stage) cp_async_wait_all();
            __syncthreads();
            // partial outputs: row i of the last matrix, columns of this block (the same warp owns row i in every block)
            for (int i0 = warp * kApRows; i0 < d; i0 += kApWarps * kApRows) {
                const int rv = min(kApRows, d - i0);
                float u[kApRows][TB];
                if (VEC && a.stage)
                    warp_dots<kApRows, TB, VEC>(wls + (size_t)i0 * nh, nh, rv, nh, as, kApHB, u);
                else
                    warp_dots<kApRows, TB, VEC>(Wl + (size_t)i0 * h + hb, h, rv, nh, as, kApHB, u);
                if (lane == 0) {
#pragma unroll
                    for (int r = 0; r < kApRows; ++r)
                        if (r < rv)
#pragma unroll
                            for (int t = 0; t < TB; ++t) up[(size_t)t * d + i0 + r] += u[r][t];
                }
            }
            __syncthreads();
        }
        // hand the partial sums to the first CTA of the cluster
        __syncwarp();
        if (t0 == 0) sm100::cluster_wait();
        for (int e = tid; e < TB * d; e += kApThreads) slot0[(size_t)rank * TB * d + e] = up[e];
        cluster.sync();
        if (rank == 0) {
            for (int e = tid; e < TB * d; e += kApThreads) {
                float s = 0.0f;
                for (int c = 0; c < CL; ++c) s += slots[(size_t)c * TB * d + e];  // fixed order
                up[e] = s;
            }
            __syncthreads();
            for (int t = warp; t < tb; t += kApWarps) {
                float* u = up + (size_t)t * d;
                warp_layernorm(u, u, d, a.eps);
                for (int i = lane; i < d; i += 32) ap_st(o, (size_t)(t0 + t) * d + i, qs[(size_t)t * d + i] + u[i]);
            }
        }
        if (t0 + TB < T) cluster.sync();  // the slots are free again (after the last pass nobody writes them any more)
    }
}

// ---- one token per sequence: the decode step -----------------------------------------------------------------------------------
// Bound by HBM (a step reads every weight once).  Every warp streams its own share of the CTA's rows through a ring of its own in
// shared memory: groups of 8 rows by bulk copies (one for the first matrices, whose rows are contiguous, 8 for column slices of
// the last), issued one ring ahead by lane 0, so 64 to 96 KB per CTA and two CTAs per SM are in flight whatever the registers hold.
// Pieces of 256 columns (or rows of more than 192 floats) leave room for one slot per warp: it is filled again once the warp has read
// it, from L2, where the prefetch at the start has brought all of the CTA's weights.  Pieces of 128 columns in three slots were slower,
// 11.7 -> 14.4 us at 94 sequences and 17.6 -> 22.3 us at 149 (GELU, d = 128, h = 512).
// The rows of the last matrix do not depend on the activations: their copies are under way while the activations are
// computed.  Eight dot products are reduced together (9 shuffles), which leaves one row per four lanes: the activation function
// runs once per row.  128 sequences x SwiGLU d = 128, h = 384 (75.5 MB): 20.9 us with loads through registers, 16.4 us.
__device__ __forceinline__ void ds_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void ds_prefetch(const void* p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
// sums of 8 values over the lanes: lane l gets the sum of v[l >> 2]
__device__ __forceinline__ float ds_reduce8(const float (&v)[8]) {
    const int lane = threadIdx.x & 31;
    float a[4], b[2];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float keep = (lane & 16) ? v[j + 4] : v[j], give = (lane & 16) ? v[j] : v[j + 4];
        a[j] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const float keep = (lane & 8) ? a[j + 2] : a[j], give = (lane & 8) ? a[j] : a[j + 2];
        b[j] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
    }
    const float keep = (lane & 4) ? b[1] : b[0], give = (lane & 4) ? b[0] : b[1];
    float c = keep + __shfl_xor_sync(0xffffffffu, give, 4);
    c += __shfl_xor_sync(0xffffffffu, c, 2);
    return c + __shfl_xor_sync(0xffffffffu, c, 1);
}

struct __align__(128) DsShared {
    uint64_t full[kDsWarps][kDsMaxSlots];
    int dead;
    float up[kDsCols];                 // this CTA's partial sums
    float slots[8 * kDsCols];          // on the first CTA: every CTA's partial sums
};
static_assert(sizeof(DsShared) == kDsFixedBytes, "");

template <typename IO, int KIND> __global__ void __launch_bounds__(kDsWarps * 32, 2) apply_stream_kernel(const ApplyArgs a) {
    constexpr int NFIRST = KIND == 0 ? 1 : 2, NMAT = NFIRST + 1;
    extern __shared__ __align__(128) unsigned char ds_smem[];
    DsShared& sh = *reinterpret_cast<DsShared*>(ds_smem);
    float* act = reinterpret_cast<float*>(ds_smem + sizeof(DsShared));  // [hidden units of the CTA, rounded up to 4]
    cg::cluster_group cluster = cg::this_cluster();
    const int CL = a.cl, seq = blockIdx.x / CL, rank = blockIdx.x % CL;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int d = a.d, h = a.h;
    const size_t dh = (size_t)d * h;
    const int per = a.per, h0 = min(h, rank * per), nh = min(h, h0 + per) - h0;
    const float* W[NMAT];
#pragma unroll
    for (int i = 0; i < NMAT; ++i) W[i] = a.W[i] + (size_t)seq * dh;
    const float* Wl = W[NFIRST];

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // Before the previous kernel of the stream is done only L2 may be touched (a prefetch has no effect on memory contents)
    if (threadIdx.x < NFIRST && nh > 0) ds_prefetch(W[threadIdx.x] + (size_t)h0 * d, (uint32_t)nh * d * 4u);
    if (nh > 0)
        for (int i = threadIdx.x; i < d; i += kDsWarps * 32) ds_prefetch(Wl + (size_t)i * h + h0, (uint32_t)nh * 4u);

    const uint32_t slot_bytes = a.slot_bytes;
    const int nslots = a.nslots;
    const uint32_t ring = sm100::smem_u32(ds_smem) + a.ring_at + (uint32_t)(warp * nslots) * slot_bytes;
    if (lane == 0)
        for (int i = 0; i < nslots; ++i) sm100::mbar_init(&sh.full[warp][i], 1);
    if (threadIdx.x == 0) sh.dead = 0;
    for (int i = threadIdx.x; i < d; i += kDsWarps * 32) sh.up[i] = 0.0f;
    sm100::fence_mbar_init();
    __syncthreads();
    sm100::cluster_arrive();  // waited for before the first store to another CTA, which has to run by then
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // this warp's groups, in order: 8 rows of every first matrix, then 8 rows x up to 256 columns of the last
    const int g1 = (nh + kDsRows - 1) / kDsRows, mine1 = warp < g1 ? (g1 - warp + kDsWarps - 1) / kDsWarps : 0;
    const int pieces = (nh + kDsCols - 1) / kDsCols, g2 = (d + kDsRows - 1) / kDsRows;
    const int mine2 = (warp < g2 ? (g2 - warp + kDsWarps - 1) / kDsWarps : 0) * pieces;
    const int total = mine1 * NFIRST + mine2;
    int issued = 0;
    auto issue = [&]() {  // the next group of the list into its slot
        const int s = issued % nslots;
        const uint32_t dst = ring + (uint32_t)s * slot_bytes, bar = sm100::smem_u32(&sh.full[warp][s]);
        if (issued < mine1 * NFIRST) {
            const int j = (warp + (issued / NFIRST) * kDsWarps) * kDsRows, rows = min(kDsRows, nh - j);
            if (lane == 0) {
                const uint32_t bytes = (uint32_t)rows * d * 4u;
                sm100::mbar_expect_tx(&sh.full[warp][s], bytes);
                ds_copy(dst, W[NFIRST == 2 ? issued % NFIRST : 0] + (size_t)(h0 + j) * d, bytes, bar);
            }
        } else {
            const int e = issued - mine1 * NFIRST, i = (warp + (e / pieces) * kDsWarps) * kDsRows, c = (e % pieces) * kDsCols;
            const int rows = min(kDsRows, d - i), cols = min(kDsCols, nh - c);
            if (lane == 0) sm100::mbar_expect_tx(&sh.full[warp][s], (uint32_t)rows * cols * 4u);
            __syncwarp();
            if (lane < rows) ds_copy(dst + (uint32_t)lane * cols * 4u, Wl + (size_t)(i + lane) * h + h0 + c, (uint32_t)cols * 4u, bar);
        }
        ++issued;
    };
    for (int i = 0; i < nslots && issued < total; ++i) issue();

    // the token: lane l holds elements 4 l .. and 128 + 4 l ..
    float4 x[2];
    const IO* q = reinterpret_cast<const IO*>(a.q) + (size_t)seq * d;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const int c = 128 * p + 4 * lane;
        x[p] = c < d ? make_float4(ap_ld<IO>(q, c), ap_ld<IO>(q, c + 1), ap_ld<IO>(q, c + 2), ap_ld<IO>(q, c + 3)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }

    int done = 0;
    // 8 dot products of the next group (row length n, a multiple of 4) with v
    auto dots = [&](int n, const float4 (&v)[2]) -> float {
        const int s = done % nslots;
        const uint32_t parity = (uint32_t)(done / nslots) & 1u;
        volatile int* dead = &sh.dead;
        if (!sm100::mbar_try_wait<false>(&sh.full[warp][s], parity) && !*dead) {  // bounded; a copy cannot fail short of a device fault
            const long long t0 = clock64();
            int spins = 0;
            while (!sm100::mbar_try_wait<false>(&sh.full[warp][s], parity))
                if ((++spins & 255) == 0 && (*dead || clock64() - t0 > sm100::kWaitCycles)) { *dead = 1; break; }
        }
        __syncwarp();
        const float* w = reinterpret_cast<const float*>(ds_smem + a.ring_at + (uint32_t)(warp * nslots + s) * slot_bytes);
        float acc[kDsRows];
#pragma unroll
        for (int r = 0; r < kDsRows; ++r) acc[r] = 0.0f;
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int c = 128 * p + 4 * lane;
            if (c < n) {
#pragma unroll
                for (int r = 0; r < kDsRows; ++r) {
                    const float4 y = *reinterpret_cast<const float4*>(w + (size_t)r * n + c);
                    acc[r] += y.x * v[p].x + y.y * v[p].y + y.z * v[p].z + y.w * v[p].w;
                }
            }
        }
        __syncwarp();  // every lane has read its part: the slot may be filled again
        ++done;
        if (issued < total) issue();
        return ds_reduce8(acc);
    };

    for (int g = 0; g < mine1; ++g) {
        const int j = (warp + g * kDsWarps) * kDsRows + (lane >> 2);
        const float z1 = dots(d, x);
        float y;
        if (KIND == 0) y = gelu_f(z1);
        else y = silu_f(z1) * dots(d, x);
        if ((lane & 3) == 0 && j < nh) act[j] = y;
    }
    __syncthreads();
    for (int g = 0; g < mine2; ++g) {
        const int i = (warp + (g / pieces) * kDsWarps) * kDsRows + (lane >> 2), c0 = (g % pieces) * kDsCols, n = min(kDsCols, nh - c0);
        float4 v[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int c = 128 * p + 4 * lane;
            v[p] = c < n ? *reinterpret_cast<const float4*>(act + c0 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const float u = dots(n, v);
        if ((lane & 3) == 0 && i < d) sh.up[i] += u;  // the same lane owns row i in every piece
    }
    __syncthreads();
    // hand the partial sums to the first CTA of the cluster
    __syncwarp();
    sm100::cluster_wait();
    // (there is no status word to report a wait that gave up: the sequence's outputs become NaN)
    const bool dead = *(volatile int*)&sh.dead;
    float* slot0 = cluster.map_shared_rank(&sh.slots[0], 0);
    for (int i = threadIdx.x; i < d; i += kDsWarps * 32) slot0[(size_t)rank * d + i] = dead ? __int_as_float(0x7fffffff) : sh.up[i];
    cluster.sync();
    if (rank == 0) {
        for (int i = threadIdx.x; i < d; i += kDsWarps * 32) {
            float s = 0.0f;
            for (int c = 0; c < CL; ++c) s += sh.slots[(size_t)c * d + i];  // fixed order
            sh.up[i] = s;
        }
        __syncthreads();
        if (warp == 0) {
            warp_layernorm(sh.up, sh.up, d, a.eps);
            IO* o = reinterpret_cast<IO*>(a.o) + (size_t)seq * d;
            for (int i = lane; i < d; i += 32) ap_st(o, (size_t)i, ap_ld<IO>(q, (size_t)i) + sh.up[i]);
        }
    }
    if (dead) {  // copies nobody waited for may still be under way to this CTA's shared memory
        const long long t0 = clock64();
        while (clock64() - t0 < 8000000) {}
    }
}

// A kernel's shared-memory limit, once per device.  The size varies from call to call; the limit is the largest of them, so that host
// threads that come here together write the same value (a limit that followed the calls could be set back by a smaller one).
template <typename K> cudaError_t allow_smem(K kernel, size_t most, std::atomic<bool> (&done)[64]) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || (dev >= 0 && dev < 64 && done[dev])) return e;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
    return e;
}

template <typename IO, int KIND> int launch_stream(const ApplyArgs& a_in, cudaStream_t st) {
    ApplyArgs a = a_in;
    const StreamGeometry g = apply_stream_geometry(a.N, a.d, a.h);
    a.cl = g.cl; a.per = g.per; a.nslots = g.nslots; a.slot_bytes = g.slot_bytes; a.ring_at = g.ring_at;
    static std::atomic<bool> done[64];
    if (cudaError_t e = allow_smem(apply_stream_kernel<IO, KIND>, kDsMaxSmem, done)) return (int)e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(a.N * a.cl));
    cfg.blockDim = dim3(kDsWarps * 32);
    cfg.dynamicSmemBytes = g.smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)a.cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see griddepcontrol in the kernel
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, apply_stream_kernel<IO, KIND>, a);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaGetLastError();
}

}  // namespace

size_t apply_smem_bytes(int d, int cl, int tb) { return ((size_t)tb * d * (2 + cl) + (size_t)tb * kApHB) * sizeof(float); }

namespace {

template <typename IO, int KIND, int TB, bool VEC>
int launch_apply(const ApplyArgs& a, cudaStream_t st) {
    const size_t smem = apply_smem_bytes(a.d, a.cl, TB) + (a.stage ? (size_t)kApStageBytes : 0);
    static std::atomic<bool> done[64];
    if (cudaError_t e = allow_smem(apply_kernel<IO, KIND, TB, VEC>, kApMaxSmem, done)) return (int)e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(a.N * a.cl));
    cfg.blockDim = dim3(kApThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)a.cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see griddepcontrol in the kernel
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, apply_kernel<IO, KIND, TB, VEC>, a);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaGetLastError();
}

template <typename IO, int KIND>
int dispatch_apply(const ApplyArgs& a, bool vec, cudaStream_t st) {
    if (a.tb == 1) return vec ? launch_apply<IO, KIND, 1, true>(a, st) : launch_apply<IO, KIND, 1, false>(a, st);
    return vec ? launch_apply<IO, KIND, 4, true>(a, st) : launch_apply<IO, KIND, 4, false>(a, st);
}

}  // namespace

int apply_token_block(int T) { return T == 1 ? 1 : 4; }

// The last matrix's block [d][min(256, hidden units per CTA)] is staged when it fits the staging buffer.
int apply_can_stage(int d, int h, int cl) {
    const int per = ((h + cl - 1) / cl + 3) & ~3;
    const int nh = per < kApHB ? per : kApHB;
    return (size_t)d * nh * sizeof(float) <= (size_t)kApStageBytes;
}

int apply_launch(const ApplyArgs& a, int kind, int io_dtype, void* stream) {
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // 16-byte loads need rows that start on 16-byte boundaries: d and h multiples of 4, 16-byte aligned bases
    bool vec = (a.d % 4 == 0) && (a.h % 4 == 0);
    const int nmat = kind == 0 ? 2 : 3;
    for (int i = 0; i < nmat; ++i) vec = vec && (reinterpret_cast<uintptr_t>(a.W[i]) % 16 == 0);
    // one token per sequence, bulk copies of whole rows: same alignment, and a token that two 16-byte pieces per lane hold
    if (vec && a.T == 1 && a.d <= kDsCols && a.h <= kDsMaxHidden) {
        if (io_dtype == 0) return kind == 0 ? launch_stream<float, 0>(a, st) : launch_stream<float, 1>(a, st);
        return kind == 0 ? launch_stream<__nv_bfloat16, 0>(a, st) : launch_stream<__nv_bfloat16, 1>(a, st);
    }
    if (io_dtype == 0)
        return kind == 0 ? dispatch_apply<float, 0>(a, vec, st) : dispatch_apply<float, 1>(a, vec, st);
    return kind == 0 ? dispatch_apply<__nv_bfloat16, 0>(a, vec, st) : dispatch_apply<__nv_bfloat16, 1>(a, vec, st);
}

}  // namespace e2ttt
