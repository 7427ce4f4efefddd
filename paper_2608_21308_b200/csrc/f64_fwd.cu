// Forward for fp32 I/O: Algorithm 1 chunk after chunk in fp64, any d, h, C and both networks.  A cluster of 1-16 CTAs per sequence, five
// phases per chunk (f64_common.cuh): activations of the keys | u of the keys, activations of the queries | rows of the keys, the next
// chunk's tokens and scalar kernels and the rows of the queries of the one before | adjoint of z, u of the queries | state transition.
// With a compact layout (f64_compact) seven: activations of both | u of both | rows of both | adjoint of z | the keys' rows times K^M |
// state transition | the next chunk's tokens.
#include "f64_common.cuh"

namespace e2ttt {

namespace {

enum { kFK, kFK1, kFU, kFQ, kFPz, kFUq, kFUpd, kFUpd1 = kFUpd + 3, kFJobs = kFUpd1 + 3 };
static_assert(kFJobs * sizeof(F64Job) <= kF64FwdTable);
struct F64Scalars {  // ChunkScalars for chunks of up to C tokens
    double *kW, *kM, *bt, *gt, *S, &cw, &cm, &cb;
    __device__ F64Scalars(double* p, int C) : kW(p), kM(p + C), bt(p + 2 * C), gt(p + 3 * C + 1), S(p + 4 * C + 2), cw(p[5 * C + 3]), cm(p[5 * C + 4]), cb(p[5 * C + 5]) {}
};

// PER_SM: CTAs per SM (f64_fwd_two)
template <int PER_SM> __global__ void __launch_bounds__(kF64Threads, PER_SM) f64_fwd_kernel(const SimtFwdArgs a, const int sw, const unsigned table) {
    extern __shared__ __align__(16) unsigned char f64_smem[];
    F64Job* const job = reinterpret_cast<F64Job*>(f64_smem + table);
    double* const sc0 = reinterpret_cast<double*>(f64_smem + table + kF64FwdTable);  // scalar kernels, by the chunk's parity
    const int CL = a.cl, seq = blockIdx.x / CL, rank = blockIdx.x % CL;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int NMAT = sw ? 3 : 2, LAST = NMAT - 1;
    const int d = a.d, h = a.h, C = a.C, L = a.L;
    const size_t dh = (size_t)d * h;
    const SimtLayout& lay = a.lay;
    const F64Layout& fl = lay.fl;
    double* ws = reinterpret_cast<double*>(a.ws) + (size_t)seq * lay.per_seq;
    const float* q = reinterpret_cast<const float*>(a.q) + (size_t)seq * a.Ls * d;
    const float* k = reinterpret_cast<const float*>(a.k) + (size_t)seq * a.Ls * d;
    const float* v = reinterpret_cast<const float*>(a.v) + (size_t)seq * a.Ls * d;
    float* o = reinterpret_cast<float*>(a.o) + (size_t)seq * a.Ls * d;
    const float* eta = a.eta + (size_t)seq * a.Ls;
    const float* beta = a.beta + (size_t)seq * a.Ls;
    const float* gamma = a.gamma + (size_t)seq * a.Ls;
    const int parts = f64_parts(C, d, h);
    const size_t pstride = (size_t)C * d;
    const bool normed = a.row_norm[0] != nullptr, compact = fl.compact;
    const size_t state_bytes = (size_t)2 * NMAT * dh * sizeof(double);
    double* saved = ws + (a.save_states == 2 ? lay.cck : lay.ckpt);
    // The last chunk's transition writes the final state itself, a pass over the state less.  With the table below built by all warps: one
    // token, d = 128, h = 512, one sequence 88.3 -> 84.3 us, 64 sequences 610 -> 581.
    const bool direct = !normed && a.W_final[0];

    for (int i = 0; i < NMAT; ++i) {  // i-th matrix: state, and the first slot of the saved ones
        struct WM { double w, m; };
        const double* ck = a.init_slot >= 0 ? ws + lay.cck + (size_t)a.init_slot * 2 * NMAT * dh : nullptr;  // a segment of the recomputation
        const float* wi = a.W_init[i] + (size_t)seq * dh;
        const float* mi = a.M_init[i] ? a.M_init[i] + (size_t)seq * dh : nullptr;
        auto put = [&](size_t e, const WM& x) {
            ws[lay.W[i] + e] = x.w;
            ws[lay.M[i] + e] = x.m;
            if (a.save_states) { saved[(size_t)i * dh + e] = x.w; saved[(size_t)(NMAT + i) * dh + e] = x.m; }
        };
        if (ck)
            batched_for<8>(tid + (size_t)rank * kF64Threads, dh, (size_t)kF64Threads * CL,
                           [&](size_t e) { return WM{ck[(size_t)i * dh + e], ck[(size_t)(NMAT + i) * dh + e]}; }, put);
        else  // converted when stored, so that all loads of a batch are in flight: the 64 sequences above 573 -> 452 us
            batched_for<16>(tid + (size_t)rank * kF64Threads, dh, (size_t)kF64Threads * CL, [&](size_t e) { return float2{wi[e], mi ? mi[e] : 0.0f}; },
                            [&](size_t e, const float2& x) { put(e, WM{(double)x.x, (double)x.y}); });
    }
    // a chunk's tokens -> fp64, for the products
    auto tokens = [&](int c) {
        const size_t e0 = (size_t)c * C * d, n = (size_t)min(C, L - c * C) * d;
        double *kt = ws + fl.fK[c & 1], *qt = ws + fl.fQ;
        for (size_t e = tid + (size_t)rank * kF64Threads; e < n; e += (size_t)kF64Threads * CL) {
            kt[e] = (double)k[e0 + e];
            qt[e] = (double)q[e0 + e];
        }
    };
    auto scalars = [&](int c) {  // Algorithm 1 line 2: scalar kernels and carries; one warp, beside the rows of the chunk before
        F64Scalars sc(sc0 + (c & 1) * (5 * C + 8), C);
        if (warp == kF64Warps - 1) chunk_scalars_warp<double>(eta + c * C, beta + c * C, gamma + c * C, min(C, L - c * C), &sc);
    };
    tokens(0);
    scalars(0);
    {  // the table, a job per warp at a time
        auto mine = [&](int j) { return lane == 0 && warp == j % (kF64Warps - 1); };  // (the last warp has the scalar kernels)
        const double* W = ws + lay.W[0];
        const double* Wl = ws + lay.W[LAST];
        auto act = [&](F64Job& j, size_t x, size_t out) {
            f64_make(j, kEpiAct, h, -1 - C, NMAT - 1, 1, 1, h, sw);
            f64_seg(j, d, f64_op(W, d, 1), f64_op(ws + x, d, 1));
            if (sw) f64_a(j, 1, f64_op(ws + lay.W[1], d, 1));
            f64_out(j, 0, f64_ptr(ws + out));
        };
        for (int b = 0; b < 2; ++b) {  // by the chunk's parity
            if (!mine(b ? kFK1 : kFK)) continue;
            F64Job& j = job[b ? kFK1 : kFK];
            act(j, fl.fK[b], fl.fA);
            f64_out(j, 1, f64_ptr(ws + fl.fc1));
            if (sw) f64_out(j, 2, f64_ptr(ws + fl.fc2));
        }
        if (mine(kFQ)) act(job[kFQ], fl.fQ, fl.fAq);
        auto to_u = [&](F64Job& j, size_t x, size_t out) {
            f64_make(j, kEpiStore, d, -1 - C, 1, 1, 1, d, sw, parts);
            f64_seg(j, h, f64_op(Wl, h, 1), f64_op(ws + x, h, 1));
            f64_out(j, 0, f64_ptr(ws + out));
            j.pstride = (long long)pstride;
        };
        if (mine(kFU)) to_u(job[kFU], fl.fA, fl.fUk);
        if (mine(kFUq)) to_u(job[kFUq], fl.fAq, fl.fUq);
        if (mine(kFPz)) {
            F64Job& j = f64_make(job[kFPz], kEpiPz, h, -1 - C, 1, 1, 1, h, sw);
            f64_seg(j, d, f64_op(Wl, 1, h), f64_op(ws + fl.fPu, d, 1));
            for (int i = 0; i < LAST; ++i) {
                f64_pre(j, f64_ptr(ws + (i ? fl.fc2 : fl.fc1)));
                f64_out(j, 4 + 2 * i, f64_ptr(ws + fl.fPzW[i]));
                f64_out(j, 5 + 2 * i, f64_ptr(ws + fl.fPzM[i]));
            }
        }
        // both weighted aggregations of every matrix, fused with the state transition
        for (int b = 0; b < 2; ++b)
            for (int i = 0; i < NMAT; ++i) {
                if (!mine((b ? kFUpd1 : kFUpd) + i)) continue;
                const int rows = i == LAST ? d : h, cols = i == LAST ? h : d;
                F64Job& j = f64_make(job[(b ? kFUpd1 : kFUpd) + i], kEpiUpdate, rows, cols, 2, 0, cols, 1, sw);
                f64_seg(j, -1, f64_op(ws + (i == LAST ? fl.fPuW : fl.fPzW[i]), 1, rows), f64_op(ws + (i == LAST ? fl.fA : fl.fK[b]), 1, cols));
                f64_a(j, 1, f64_op(ws + (i == LAST ? fl.fPuM : fl.fPzM[i]), 1, rows));
                f64_inout(j, 0, f64_ptr(ws + lay.W[i]));
                f64_inout(j, 1, f64_ptr(ws + lay.M[i]));
                f64_out(j, 2, normed ? F64Ptr{nullptr, 0} : f64_ptr(saved + (size_t)i * dh));  // (normalised first: saved there)
                f64_out(j, 3, f64_ptr(saved + (size_t)(NMAT + i) * dh));
                if (direct) {  // (floats)
                    f64_out(j, 4, f64_ptr(reinterpret_cast<double*>(a.W_final[i] + (size_t)seq * dh)));
                    f64_out(j, 5, f64_ptr(reinterpret_cast<double*>(a.M_final[i] + (size_t)seq * dh)));
                }
            }
    }
    __syncthreads();
    phase_sync(CL);

    auto u_row = [&](size_t up, int m, int i) { return f64_parts_at(ws + up, (size_t)m * d + i, parts, pstride); };
    const double inv = 1.0 / d;
    auto output_row = [&](int c, int m) {  // o = q + LN(u)
        const size_t row = ((size_t)c * C + m) * d;
        double su = 0.0;
#pragma unroll 2
        for (int i = lane; i < d; i += 32) su += u_row(fl.fUq, m, i);
        const double mu = warp_sum(su) * inv;
        double var = 0.0;
#pragma unroll 2
        for (int i = lane; i < d; i += 32) { const double x = u_row(fl.fUq, m, i) - mu; var += x * x; }
        const double r = r_rsqrt(warp_sum(var) * inv + (double)a.eps);
#pragma unroll 2
        for (int i = lane; i < d; i += 32) o[row + i] = (float)((double)q[row + i] + (u_row(fl.fUq, m, i) - mu) * r);
    };
    F64Ctx cx{};
    for (int c = 0; c < a.nchunks; ++c) {
        const int s = c * C, len = min(C, L - s);
        const float* kc = k + (size_t)s * d;
        const float* vc = v + (size_t)s * d;
        const F64Scalars sc(sc0 + (c & 1) * (5 * C + 8), C);
        cx.len = len;
        cx.kW = sc.kW; cx.kM = sc.kM; cx.cw = sc.cw; cx.cm = sc.cm; cx.cb = sc.cb;
        auto run = [&](int j0, int j1) { f64_jobs<PER_SM == 2 ? kF64FwdSmall : kF64Fwd>(job, j0, j1, cx, rank, CL, f64_smem); };

        // Algorithm 1 line 1: the network, keys first
        const int odd = c & 1;
        run(kFK + odd, kFK + odd + 1);
        if (compact) run(kFQ, kFQ + 1);
        phase_sync(CL);
        run(kFU, a.o && !compact ? kFQ + 1 : kFQ);
        if (compact) run(kFUq, kFUq + 1);
        phase_sync(CL);
        // Algorithm 1 line 3: layer norm, e = f(k) - v and pu = dL/du for the key rows; tokens and scalars of the next chunk
        if (c + 1 < a.nchunks) {
            if (!compact) tokens(c + 1);
            scalars(c + 1);
        }
        for (int m = rank + CL * warp; m < len + (a.o && c > 0 && !compact ? C : 0); m += CL * kF64Warps) {
            if (m >= len) {  // rows of the queries of the chunk before
                output_row(c - 1, m - len);
                continue;
            }
            if (compact) output_row(c, m);  // (a lane writes pu where it alone read u of the query)
            double su = 0.0;
            double* pu = ws + fl.fPu + (size_t)m * d;
#pragma unroll 2
            for (int i = lane; i < d; i += 32) { const double x = u_row(fl.fUk, m, i); pu[i] = x; su += x; }
            const double mu = warp_sum(su) * inv;
            double var = 0.0;
#pragma unroll 2
            for (int i = lane; i < d; i += 32) { const double x = pu[i] - mu; var += x * x; }
            const double r = r_rsqrt(warp_sum(var) * inv + (double)a.eps);
            double se = 0.0, sey = 0.0;
#pragma unroll 2
            for (int i = lane; i < d; i += 32) {
                const double y = (pu[i] - mu) * r, e = (double)kc[(size_t)m * d + i] + y - (double)vc[(size_t)m * d + i];
                se += e;
                sey += e * y;
            }
            se = warp_sum(se) * inv;
            sey = warp_sum(sey) * inv;
#pragma unroll 2
            for (int i = lane; i < d; i += 32) {
                const double y = (pu[i] - mu) * r, e = (double)kc[(size_t)m * d + i] + y - (double)vc[(size_t)m * d + i];
                const double x = r * (e - se - y * sey);
                pu[i] = x;
                ws[fl.fPuW + (size_t)m * d + i] = x * sc.kW[m];
                if (!compact) ws[fl.fPuM + (size_t)m * d + i] = x * sc.kM[m];
            }
        }
        phase_sync(CL);
        // back through the last matrix and the activation
        run(kFPz, a.o && !compact ? kFUq + 1 : kFUq);
        phase_sync(CL);
        if (compact) {
            for (int m = rank + CL * warp; m < len; m += CL * kF64Warps) {
                double* pu = ws + fl.fPu + (size_t)m * d;
#pragma unroll 4
                for (int i = lane; i < d; i += 32) pu[i] *= sc.kM[m];
            }
            phase_sync(CL);
        }
        // Algorithm 1 lines 4-7
        int slot = -1;  // the saved state that this chunk's end is
        if (a.save_states == 1 && (c + 1 < a.nchunks || normed)) slot = c + 1;
        else if (a.save_states == 2 && c + 1 < a.nchunks && (c + 1) % lay.seg == 0) slot = (c + 1) / lay.seg;
        cx.save = slot < 0 ? -1 : (long long)(slot * state_bytes);
        cx.last = direct && c + 1 == a.nchunks;
        run(odd ? kFUpd1 : kFUpd, (odd ? kFUpd1 : kFUpd) + NMAT);
        if (cx.last) break;  // (nothing that follows reads it)
        phase_sync(CL);
        if (compact && c + 1 < a.nchunks) {
            tokens(c + 1);
            phase_sync(CL);
        }
        // post-chunk normalisation (optional): every row w of every W_i becomes n w / (||w|| + eps_n); one warp per row
        if (normed) {
            const int maxdim = d > h ? d : h;
            for (int i = 0; i < NMAT; ++i) {
                const int rows = (i == LAST) ? d : h, cols = (i == LAST) ? h : d;
                const float* target = a.row_norm[i] + (size_t)seq * rows;
                for (int r = warp + rank * kF64Warps; r < rows; r += kF64Warps * CL) {
                    double* w = ws + lay.W[i] + (size_t)r * cols;
                    double ss = 0.0;
#pragma unroll 2
                    for (int j = lane; j < cols; j += 32) ss += w[j] * w[j];
                    const double nrm = sqrt(warp_sum(ss));
                    const double f = (double)target[r] / (nrm + (double)a.norm_eps);
                    double* to = slot >= 0 ? saved + (size_t)slot * 2 * NMAT * dh + (size_t)i * dh + (size_t)r * cols : nullptr;
#pragma unroll 2
                    for (int j = lane; j < cols; j += 32) {
                        const double x = w[j] * f;
                        w[j] = x;
                        if (to) to[j] = x;
                    }
                    if (a.save_states && lane == 0) ws[lay.rown + ((size_t)c * 3 + i) * maxdim + r] = nrm;
                }
            }
            phase_sync(CL);
        }
    }
    if (a.o && !compact)
        for (int m = rank + CL * warp; m < L - (a.nchunks - 1) * C; m += CL * kF64Warps) output_row(a.nchunks - 1, m);
    for (int i = 0; i < NMAT; ++i) {
        if (direct || !a.W_final[i]) continue;  // none: recomputation for the reverse pass, only the saved states matter
        float* wf = a.W_final[i] + (size_t)seq * dh;
        float* mf = a.M_final[i] + (size_t)seq * dh;
        struct WM { double w, m; };
        batched_for<8>(tid + (size_t)rank * kF64Threads, dh, (size_t)kF64Threads * CL,
                       [&](size_t e) { return WM{ws[lay.W[i] + e], ws[lay.M[i] + e]}; },
                       [&](size_t e, const WM& x) { wf[e] = (float)x.w; mf[e] = (float)x.m; });
    }
}

}  // namespace

int f64_fwd_launch(const SimtFwdArgs& a, int kind, void* stream) {
    static std::atomic<int> state[2][64];
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const int sw = kind == 0 ? 0 : 1;
    const size_t sc = f64_fwd_scalars(a.C);
    constexpr size_t most = kF64FwdTile + kF64FwdTable + f64_fwd_scalars(kMaxC);
    static_assert(most <= 232448, "227 KB of shared memory per CTA");
    if (f64_fwd_two(a.N, a.d, a.h, a.C)) {
        const size_t smem = f64_fwd_small(a.d, a.h, a.C);
        return simt_launch(f64_fwd_kernel<2>, a, kF64Threads, smem, 113 << 10, state[0], st, sw, (unsigned)(smem - kF64FwdTable - sc));
    }
    return simt_launch(f64_fwd_kernel<1>, a, kF64Threads, kF64FwdTile + kF64FwdTable + sc, most, state[1], st, sw, (unsigned)kF64FwdTile);
}

}  // namespace e2ttt
