// Building blocks of the fp64 kernels (fp32 I/O: the checking mode), f64_fwd.cu and f64_bwd.cu.
//
// What bounds a small problem: one sequence's chunks are a chain of short phases, and a phase of a cluster of 16 CTAs has no more to
// do than an L2 round trip takes.  So a phase must cost little more than that: few phases (every product that is ready runs in the
// same one), and little code.  With each product's loaders and epilogue inlined the reverse pass was 800 KB of machine code, walked
// once per chunk: its phases waited for instructions, 6 us each.  Here a product is data - operands with strides, an epilogue number -
// built once per launch in shared memory, and all products of a chunk go through the same few instantiations of f64_units(): 16 chunks
// of 16 tokens, d = 64, h = 256, one sequence, forward and reverse pass 2806 -> 948 us.
//
// A result does not depend on the cluster's size: tilings, the parts a contraction is cut into and all orders of summation follow from
// the shape alone.
#pragma once
#include "simt_common.cuh"
#include "simt_layout.h"

namespace e2ttt {

constexpr int kF64Threads = 256, kF64Warps = kF64Threads / 32;

// Where an operand or a result of a job lies: for the chunk at hand p, a chunk later p + step (bytes)
struct F64Ptr {
    double* p;
    long long step;
};
struct F64Op {  // element (r, k): p[r * rs + k * ks]; one of rs, ks is 1
    F64Ptr at;
    int rs, ks;
};
// out(m, n) = sum over segments and k of a_i(m, k) b(n, k), for `na` operands a_i on one b.  Dimensions of -1: tokens of the chunk
enum F64Epi { kEpiStore, kEpiAct, kEpiPz, kEpiUpdate, kEpiDq, kEpiXY, kEpiZ, kEpiT };
constexpr int kF64Segs = 4, kF64Pre = 20, kF64Out = 26, kF64Aux = 34, kF64Ptrs = 35;
struct F64Job {
    int M, N, nseg, na, epi, wide, parts, mfast, npre;
    int om, on;         // element (m, n) of every pre / out array is number m * om + n * on
    int sw;             // SwiGLU
    int auxn;
    long long pstride;  // elements between the parts of a result
    F64Ptr ptr[kF64Ptrs];  // operands 5 s + i (i-th a of segment s), 5 s + 4 (b); what results combine with; results
    int rs[kF64Segs * 5], ks[kF64Segs * 5], K[kF64Segs];
};
struct F64Ctx {
    int len;
    double cw, cm, cb;
    const double *kW, *kM;  // shared memory
    long long save;         // kEpiUpdate: bytes from results 2, 3 to the slot that takes the new state, -1: none
    bool last;              // kEpiUpdate: the new state is the call's result: to 4, 5 (floats) instead of 0, 1
};

// Staging of one product: two stages.  Rows of ROW doubles per k: the fragments' loads (4 k x 4 neighbouring rows a half-warp) are free of
// bank conflicts at ROW = 4 mod 16.  Four operands run in 16 x 16 tiles only.  MODE: whose products, and with kF64FwdSmall (two CTAs on an SM) a
// unit's sums lie over the slice that was multiplied last, a barrier later.
enum { kF64Bwd, kF64Fwd, kF64FwdSmall };
template <int NA, int T, int MODE> struct F64Smem {
    static constexpr bool SMALL = MODE == kF64FwdSmall;
    static constexpr int KS = T == 16 ? 64 : 32, SPLIT = T == 16 ? 2 : 1, ROW = T + 4;
    static constexpr int PRE = SMALL ? 2 : NA == 4 ? 6 : 4;
    double a[2][NA + 1][KS][ROW];  // b is the last
    double sums[SMALL ? 1 : NA * SPLIT][SMALL ? 1 : T * T];
    double pre[2][PRE][T * T];
    __device__ __forceinline__ double* part(int stage, int i) { return SMALL ? &a[stage][0][0][0] + i * (T * T) : sums[i]; }
    static_assert(!SMALL || NA * SPLIT * T * T <= (NA + 1) * KS * ROW);
};
constexpr size_t kF64TileSmem = sizeof(F64Smem<4, 16, kF64Bwd>) > sizeof(F64Smem<2, 32, kF64Bwd>) ? sizeof(F64Smem<4, 16, kF64Bwd>) : sizeof(F64Smem<2, 32, kF64Bwd>);
static_assert(sizeof(F64Smem<2, 32, kF64Fwd>) <= kF64FwdTile && sizeof(F64Smem<2, 32, kF64FwdSmall>) <= f64_small_tile(true) && sizeof(F64Smem<2, 16, kF64FwdSmall>) <= f64_small_tile(false));

__device__ __forceinline__ void f64_copy(uint32_t dst, const void* src, bool in) {  // 8 bytes; zeros where !in
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(in ? 8 : 0) : "memory");
}
// 8 x 8 += (8 x 4) (4 x 8).  A lane's a: row lane / 4, k lane % 4; b: column lane / 4; c: row lane / 4, columns 2 (lane % 4), + 1
__device__ __forceinline__ void f64_mma(double (&c)[2], double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};" : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}
__device__ __forceinline__ int f64_div(int x, int y) {  // x < 2^21
    return y == 1 ? x : (int)__fdividef((float)x + 0.5f, (float)y);
}

// a = act(z), its derivatives as the epilogues use them.  GELU: f1 = gelu', f3 = gelu''.  SwiGLU: f1 = z2 silu'(z1), f2 = silu(z1),
// f3 = z2 silu''(z1), f4 = silu'(z1).
struct F64Act {
    double a, f1, f2, f3, f4;
};
static __device__ __noinline__ F64Act f64_act(int sw, int deriv, double z1, double z2) {
    F64Act o;
    if (!sw) {
        const double cdf = norm_cdf(z1), pdf = deriv ? norm_pdf(z1) : 0.0;
        o.a = z1 * cdf;
        o.f1 = cdf + z1 * pdf;
        o.f2 = 0.0;
        o.f3 = pdf * (2.0 - z1 * z1);
        o.f4 = 0.0;
    } else {
        const double s = sigmoid_f(z1), g = s * (1.0 + z1 * (1.0 - s));
        o.a = z1 * s * z2;
        o.f1 = z2 * g;
        o.f2 = z1 * s;
        o.f3 = z2 * s * (1.0 - s) * (2.0 + z1 * (1.0 - 2.0 * s));
        o.f4 = g;
    }
    return o;
}

// The units (tile, part of the contraction) first, first + step, .. of a job.  T = 16: 64-deep slices cut in two inside the CTA;
// T = 32: 32-deep slices.  The next slice is on its way (cp.async: no register holds it) while one is multiplied, by fp64 MMAs: they run
// no faster than FMAs, but a shared-memory access feeds four times as many products (2 x 2 FMAs per thread took 70 cycles for each of
// the 16 steps of a slice, all of it the port of shared memory).
template <int NA, int T, int MODE> static __device__ __noinline__ void f64_units(const F64Job& jb, const F64Ctx& cx, int first, int step, unsigned char* smem) {
    using S = F64Smem<NA, T, MODE>;
    constexpr int KS = S::KS, SPLIT = S::SPLIT, PER = T * KS / kF64Threads, EL = T * T / kF64Threads;
    constexpr int NT = T == 16 ? 1 : 2;  // 8 x 8 tiles per warp, below one another
    S& sm = *reinterpret_cast<S*>(smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int M = jb.M < 0 ? cx.len : jb.M, N = jb.N < 0 ? cx.len : jb.N;
    const int tn = (N + T - 1) / T, parts = jb.parts, units = tn * ((M + T - 1) / T) * parts;
    const int nseg = jb.nseg, mf = jb.mfast, epi = jb.epi, om = jb.om, on = jb.on, npre = jb.npre;
    auto seg_k = [&](int s) { const int K = jb.K[s]; return K < 0 ? cx.len : K; };
    int slices = 0;
#pragma unroll 1
    for (int s = 0; s < nseg; ++s) slices += (seg_k(s) + KS - 1) / KS;
    // this warp's tiles and its half of a slice
    const int wm = T == 16 ? (warp & 1) * 8 : (warp & 1) * 16, wn = T == 16 ? (warp >> 1 & 1) * 8 : (warp >> 1) * 8, wk = T == 16 ? warp >> 2 : 0;
    auto em = [&](int e) { return mf ? (tid + e * kF64Threads) % T : (tid + e * kF64Threads) / T; };
    auto en = [&](int e) { return mf ? (tid + e * kF64Threads) / T : (tid + e * kF64Threads) % T; };
    double acc[NA][NT][2];

    // u, m0, n0, left, seg, k0: the next slice to fetch
    int u = first, left = 0, m0 = 0, n0 = 0, seg = 0, k0 = 0;
    if (u >= units) return;
    int cu = 0, cm0 = 0, cn0 = 0, terms = 0;  // the slice being multiplied
    bool opens = true, closes = false;
#pragma unroll 1
    for (int it = -1;; ++it) {
        const int st = (it + 1) & 1;  // stage of the slice to fetch
        if (it >= 0) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
        }
        const bool more = u < units;
        const int mu = cu, mm0 = cm0, mn0 = cn0, mterms = terms;
        const bool mopens = opens, mcloses = closes;
        if (more) {
            opens = left == 0;
            if (opens) {
                const int tile = f64_div(u, parts), part = u - tile * parts, tm = f64_div(tile, tn);
                m0 = tm * T;
                n0 = (tile - tm * tn) * T;
                int s0 = f64_div(part * slices, parts);
                left = f64_div((part + 1) * slices, parts) - s0;
                for (seg = 0; seg < nseg - 1; ++seg) {
                    const int ns = (seg_k(seg) + KS - 1) / KS;
                    if (s0 < ns) break;
                    s0 -= ns;
                }
                k0 = s0 * KS;
            }
            const int K = seg_k(seg);
#pragma unroll
            for (int a = 0; a <= NA; ++a) {
                const int o = 5 * seg + (a < NA ? a : 4);
                const int R = a < NA ? M - m0 : N - n0, ks = jb.ks[o], rs = jb.rs[o];
                const bool kf = ks == 1;  // neighbouring threads, neighbouring words
                int r = kf ? tid / KS : tid % T, k = kf ? tid % KS : tid / T;
                const int dr = kf ? kF64Threads / KS : 0, dk = kf ? 0 : kF64Threads / T;
                const double* base = jb.ptr[o].p;
                const double* p = base + (size_t)((a < NA ? m0 : n0) + r) * rs + (size_t)(k0 + k) * ks;
                uint32_t dst = (uint32_t)__cvta_generic_to_shared(&sm.a[st][a][k][r]);
#pragma unroll
                for (int i = 0; i < PER; ++i) {
                    const bool in = r < R && k0 + k < K;
                    f64_copy(dst, in ? p : base, in);
                    r += dr;
                    k += dk;
                    p += dr * rs + dk * ks;
                    dst += (dk * S::ROW + dr) * 8;
                }
            }
            cu = u; cm0 = m0; cn0 = n0;
            terms = min(KS, K - k0);
            closes = --left == 0;
            if (closes) {  // what the unit's results combine with
#pragma unroll
                for (int e = 0; e < EL; ++e) {
                    const int m = m0 + em(e), n = n0 + en(e);
                    const bool in = m < M && n < N;
                    const size_t off = in ? (size_t)m * om + (size_t)n * on : 0;
                    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&sm.pre[st][0][tid + e * kF64Threads]);
#pragma unroll 2
                    for (int q = 0; q < npre; ++q) f64_copy(dst + q * (T * T * 8), jb.ptr[kF64Pre + q].p + off, in);
                }
                u += step;
            } else {
                k0 += KS;
                if (k0 >= K) { k0 = 0; ++seg; }
            }
        }
        if (it < 0) continue;
        if (mopens)
#pragma unroll
            for (int a = 0; a < NA; ++a)
#pragma unroll
                for (int t = 0; t < NT; ++t) acc[a][t][0] = acc[a][t][1] = 0.0;
        const int ms = st ^ 1;
        {
            const double* pb = &sm.a[ms][NA][lane & 3][wn + (lane >> 2)];
            const double* pa = &sm.a[ms][0][lane & 3][wm + (lane >> 2)];
            const int k1 = min(mterms, (wk + 1) * (KS / SPLIT));
#pragma unroll 4
            for (int k = wk * (KS / SPLIT); k < k1; k += 4) {  // (zeros behind the last term)
                const double b = pb[k * S::ROW];
#pragma unroll
                for (int a = 0; a < NA; ++a)
#pragma unroll
                    for (int t = 0; t < NT; ++t) f64_mma(acc[a][t], pa[a * (KS * S::ROW) + k * S::ROW + 8 * t], b);
            }
        }
        if (mcloses) {
            if (S::SMALL) __syncthreads();
#pragma unroll
            for (int a = 0; a < NA; ++a)
#pragma unroll
                for (int t = 0; t < NT; ++t)
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int m = wm + 8 * t + (lane >> 2), n = wn + 2 * (lane & 3) + j;
                        sm.part(ms, a * SPLIT + wk)[mf ? n * T + m : m * T + n] = acc[a][t][j];
                    }
            __syncthreads();
            // x(e, a): result of element e; P(e, i): what it combines with; put(e, i, v): result i
            auto x = [&](int e, int a) {
                double s = sm.part(ms, a * SPLIT)[tid + e * kF64Threads];
                if (SPLIT == 2) s += sm.part(ms, a * SPLIT + 1)[tid + e * kF64Threads];
                return s;
            };
            auto P = [&](int e, int i) { return sm.pre[ms][i][tid + e * kF64Threads]; };
            auto off = [&](int e) { return (size_t)(mm0 + em(e)) * om + (size_t)(mn0 + en(e)) * on; };
            auto in = [&](int e) { return mm0 + em(e) < M && mn0 + en(e) < N; };
            auto out = [&](int i) { return jb.ptr[kF64Out + i].p; };
            if (epi == kEpiStore) {
                const long long po = (mu - f64_div(mu, parts) * parts) * jb.pstride;
#pragma unroll
                for (int a = 0; a < (NA > 2 ? 2 : NA); ++a)
#pragma unroll
                    for (int e = 0; e < EL; ++e)
                        if (in(e)) out(a)[off(e) + po] = x(e, a);
            } else if (NA <= 2 && epi == kEpiAct) {
#pragma unroll 1
                for (int e = 0; e < EL; ++e) {
                    const F64Act o = f64_act(jb.sw, out(1) != nullptr, x(e, 0), x(e, NA - 1));
                    if (!in(e)) continue;
                    const size_t f = off(e);
                    out(0)[f] = o.a;
                    if (out(1)) out(1)[f] = o.f1;
                    if (out(2)) out(2)[f] = o.f2;
                    if (out(3)) out(3)[f] = o.f3;
                    if (out(4)) out(4)[f] = o.f4;
                }
            }
            if constexpr (NA == 1) {
                if (epi == kEpiPz) {  // ph -> pz (or the adjoint of z, query rows), also times K^W, K^M; the second-order factors
#pragma unroll 1
                    for (int i = 0; i < npre; ++i) {
                        double *o = out(i), *ow = i < 2 ? out(4 + 2 * i) : nullptr, *om_ = i < 2 ? out(5 + 2 * i) : nullptr;
#pragma unroll
                        for (int e = 0; e < EL; ++e) {
                            const double v = x(e, 0) * P(e, i);
                            const int n = mn0 + en(e);
                            if (!in(e)) continue;
                            if (o) o[off(e)] = v;
                            if (ow) {
                                ow[off(e)] = v * cx.kW[n];
                                om_[off(e)] = v * cx.kM[n];
                            }
                        }
                    }
                } else if (MODE == kF64Bwd && epi == kEpiDq) {  // dq = d_o + ..
                    float* o = reinterpret_cast<float*>(out(0));
                    const float* y = reinterpret_cast<const float*>(jb.ptr[kF64Aux].p);
#pragma unroll
                    for (int e = 0; e < EL; ++e)
                        if (in(e)) o[off(e)] = (float)((double)y[off(e)] + x(e, 0));
                } else if (MODE == kF64Bwd && epi == kEpiZ) {  // adjoint of z: what came through pz, and through the hidden activation (x is minus its adjoint)
#pragma unroll 1
                    for (int i = 0; i < npre; i += 2) {
                        double* o = out(i / 2);
#pragma unroll
                        for (int e = 0; e < EL; ++e)
                            if (in(e)) o[off(e)] = P(e, i) - x(e, 0) * P(e, i + 1);
                    }
                } else if (MODE == kF64Bwd && epi == kEpiT) {  // p: T, S, W, M of the chunk's start; the carries' adjoints
                    double d0 = 0.0, d1 = 0.0, d2 = 0.0;
                    double *ot = out(0), *os = out(1);
#pragma unroll
                    for (int e = 0; e < EL; ++e)
                        if (in(e)) {
                            const double t = P(e, 0), s = P(e, 1);
                            d0 += t * P(e, 2);
                            d1 += t * P(e, 3);
                            d2 += s * P(e, 3);
                            ot[off(e)] = cx.cw * t + x(e, 0);
                            os[off(e)] = cx.cm * t + cx.cb * s;
                        }
                    d0 = warp_sum(d0); d1 = warp_sum(d1); d2 = warp_sum(d2);
                    if (lane == 0) {
                        double* q = jb.ptr[kF64Aux].p + ((size_t)mu * kF64Warps + warp) * 3;
                        q[0] = d0; q[1] = d1; q[2] = d2;
                    }
                }
            }
            if constexpr (NA == 2 && MODE != kF64Bwd) {
                if (epi == kEpiUpdate) {  // the state transition; G_t = -grad: the aggregations enter with a minus sign
                    double *ow = out(0), *om_ = out(1), *sw = nullptr, *sm_ = nullptr;
                    if (cx.save >= 0) {
                        if (out(2)) sw = reinterpret_cast<double*>(reinterpret_cast<char*>(out(2)) + cx.save);
                        sm_ = reinterpret_cast<double*>(reinterpret_cast<char*>(out(3)) + cx.save);
                    }
#pragma unroll
                    for (int e = 0; e < EL; ++e)
                        if (in(e)) {
                            const double w = cx.cw * P(e, 0) + cx.cm * P(e, 1) - x(e, 0), mm = cx.cb * P(e, 1) - x(e, 1);
                            if (cx.last) {
                                reinterpret_cast<float*>(out(4))[off(e)] = (float)w;
                                reinterpret_cast<float*>(out(5))[off(e)] = (float)mm;
                            } else {
                                ow[off(e)] = w;
                                om_[off(e)] = mm;
                            }
                            if (sw) sw[off(e)] = w;
                            if (sm_) sm_[off(e)] = mm;
                        }
                }
            }
            if constexpr (NA >= 2 && MODE == kF64Bwd) {
                if (epi == kEpiXY) {  // x = T k, y = S k (first matrices): adjoint of pz, through pz = ph act'(z) to those of ph and z
                    // p: pz1, f1, ph f3 (, pz2, f2, ph f4)
#pragma unroll
                    for (int e = 0; e < EL; ++e) {
                        double sw = 0.0, sm_ = 0.0;
                        const int m = mm0 + em(e), n = mn0 + en(e);
                        if (in(e)) {
                            const double kw = cx.kW[n], km = cx.kM[n], x0 = x(e, 0), x1 = x(e, 1), b1 = -(kw * x0 + km * x1);
                            sw = P(e, 0) * x0;
                            sm_ = P(e, 0) * x1;
                            double hb = b1 * P(e, 1), zb = b1 * P(e, 2);
                            if constexpr (NA == 4) {
                                const double x2 = x(e, 2), x3 = x(e, 3), b2 = -(kw * x2 + km * x3);
                                sw += P(e, 3) * x2;
                                sm_ += P(e, 3) * x3;
                                hb += b2 * P(e, 4);
                                zb += b2 * P(e, 5);
                                out(2)[off(e)] = b1 * P(e, 5);
                            }
                            out(0)[off(e)] = hb;
                            out(1)[off(e)] = zb;
                        }
                        // the tile's part of <pz_t, T k_t>, <pz_t, S k_t>: its rows are T neighbouring lanes
#pragma unroll
                        for (int o = T / 2; o > 0; o >>= 1) { sw += shfl_xor_r(sw, o); sm_ += shfl_xor_r(sm_, o); }
                        if (lane % T == 0 && n < N) {
                            double* q = jb.ptr[kF64Aux].p + (size_t)(mm0 / T) * jb.auxn + n;
                            q[0] = sw;
                            q[(size_t)((M + T - 1) / T) * jb.auxn] = sm_;
                        }
                        (void)m;
                    }
                }
            }
        }
        if (!more) break;
    }
    __syncthreads();  // the next job's copies go to the same stages
}

__device__ __forceinline__ int f64_job_units(const F64Job& jb, int len) {
    const int T = jb.wide ? 32 : 16, M = jb.M < 0 ? len : jb.M, N = jb.N < 0 ? len : jb.N;
    return ((M + T - 1) / T) * ((N + T - 1) / T) * jb.parts;
}
// Jobs [j0, j1) of one phase: their units are dealt to the cluster's CTAs in turn
template <int MODE> static __device__ void f64_jobs(const F64Job* jobs, int j0, int j1, const F64Ctx& cx, int rank, int nranks, unsigned char* smem) {
    int base = 0;
    for (int j = j0; j < j1; ++j) {
        const F64Job& jb = jobs[j];
        const int first = (rank - base % nranks + nranks) % nranks, n = f64_job_units(jb, cx.len);
        base += n;
        if (first >= n) continue;
        if (jb.wide) {
            if (jb.na == 1) f64_units<1, 32, MODE>(jb, cx, first, nranks, smem);
            else f64_units<2, 32, MODE>(jb, cx, first, nranks, smem);
        } else {
            if (jb.na == 1) f64_units<1, 16, MODE>(jb, cx, first, nranks, smem);
            else if (MODE != kF64Bwd || jb.na == 2) f64_units<2, 16, MODE>(jb, cx, first, nranks, smem);
            else f64_units<4, 16, kF64Bwd>(jb, cx, first, nranks, smem);
        }
    }
}

// Table builders (one thread)
__device__ __forceinline__ F64Ptr f64_ptr(double* p, long long step = 0) { return F64Ptr{p, step}; }
__device__ __forceinline__ F64Op f64_op(const double* p, int rs, int ks, long long step = 0) { return F64Op{{const_cast<double*>(p), step}, rs, ks}; }
// A dimension of C tokens is passed as -1 - C: the tiling follows from the full chunk, also in a shorter last one
static __device__ __noinline__ F64Job& f64_make(F64Job& j, int epi, int M, int N, int na, int mfast, int om, int on, int sw, int parts = 1) {
    j.epi = epi;
    j.M = M < 0 ? -1 : M;
    j.N = N < 0 ? -1 : N;
    j.wide = na <= 2 && f64_wide(M < 0 ? -1 - M : M, N < 0 ? -1 - N : N);
    j.nseg = 0;
    j.na = na; j.mfast = mfast; j.npre = 0; j.om = om; j.on = on; j.sw = sw; j.parts = parts;
    j.pstride = 0;
    j.auxn = 0;
    for (int i = 0; i < kF64Ptrs; ++i) j.ptr[i] = F64Ptr{nullptr, 0};
    return j;
}
static __device__ __noinline__ void f64_set(F64Job& j, int i, const F64Op& o) {
    j.ptr[i] = o.at;
    j.rs[i] = o.rs;
    j.ks[i] = o.ks;
}
__device__ __forceinline__ void f64_seg(F64Job& j, int K, const F64Op& a, const F64Op& b) {
    const int s = j.nseg++;
    j.K[s] = K;
    f64_set(j, 5 * s, a);
    f64_set(j, 5 * s + 4, b);
}
__device__ __forceinline__ void f64_a(F64Job& j, int i, const F64Op& a) { f64_set(j, 5 * (j.nseg - 1) + i, a); }  // i-th a of the last segment
__device__ __forceinline__ void f64_pre(F64Job& j, const F64Ptr& p) { j.ptr[kF64Pre + j.npre++] = p; }
__device__ __forceinline__ void f64_out(F64Job& j, int i, const F64Ptr& p) { j.ptr[kF64Out + i] = p; }
__device__ __forceinline__ void f64_inout(F64Job& j, int i, const F64Ptr& p) { f64_pre(j, p); f64_out(j, i, p); }
// All threads, at the end of a chunk: the pointers of the next one
__device__ __forceinline__ void f64_step(F64Job* jobs, int n) {
    for (int i = threadIdx.x; i < n * 64; i += kF64Threads)
        if ((i & 63) < kF64Ptrs) {
            F64Ptr& q = jobs[i >> 6].ptr[i & 63];
            if (q.step) q.p = reinterpret_cast<double*>(reinterpret_cast<char*>(q.p) + q.step);
        }
}

// sum of the parts of a [tokens x d] result at element e, in order
__device__ __forceinline__ double f64_parts_at(const double* p, size_t e, int parts, size_t stride) {
    double v[kF64Parts], s = 0.0;
#pragma unroll
    for (int i = 0; i < kF64Parts; ++i) v[i] = i < parts ? p[e + i * stride] : 0.0;
#pragma unroll
    for (int i = 0; i < kF64Parts; ++i) s += v[i];
    return s;
}

}  // namespace e2ttt
