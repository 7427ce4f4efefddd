// Forward for fp32 I/O: Algorithm 1 chunk after chunk in fp64, any d, h, C and both networks.  A cluster of 1-16 CTAs per sequence, five
// phases per chunk (f64_common.cuh): activations of the keys | u of the keys, activations of the queries | rows of the keys, the next
// chunk's tokens and scalar kernels and the rows of the queries of the one before | adjoint of z, u of the queries | state transition.
#include "f64_common.cuh"

namespace e2ttt {

namespace {

enum { kFK, kFK1, kFU, kFQ, kFPz, kFUq, kFUpd, kFUpd1 = kFUpd + 3, kFJobs = kFUpd1 + 3 };
struct F64FwdShared {
    F64Job job[kFJobs];
    ChunkScalars<double> sc[2];  // by the chunk's parity
};

__global__ void __launch_bounds__(kF64Threads, 1) f64_fwd_kernel(const SimtFwdArgs a, const int sw) {
    extern __shared__ __align__(16) unsigned char f64_smem[];
    F64FwdShared& sh = *reinterpret_cast<F64FwdShared*>(f64_smem + kF64TileSmem);
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
    const bool normed = a.row_norm[0] != nullptr;
    const size_t state_bytes = (size_t)2 * NMAT * dh * sizeof(double);
    double* saved = ws + (a.save_states == 2 ? lay.cck : lay.ckpt);

    for (int i = 0; i < NMAT; ++i) {  // i-th matrix: state, and the first slot of the saved ones
        struct WM { double w, m; };
        const double* ck = a.init_slot >= 0 ? ws + lay.cck + (size_t)a.init_slot * 2 * NMAT * dh : nullptr;  // a segment of the recomputation
        const float* wi = a.W_init[i] + (size_t)seq * dh;
        const float* mi = a.M_init[i] ? a.M_init[i] + (size_t)seq * dh : nullptr;
        batched_for<8>(tid + (size_t)rank * kF64Threads, dh, (size_t)kF64Threads * CL,
                       [&](size_t e) {
                           if (ck) return WM{ck[(size_t)i * dh + e], ck[(size_t)(NMAT + i) * dh + e]};
                           return WM{(double)wi[e], mi ? (double)mi[e] : 0.0};
                       },
                       [&](size_t e, const WM& x) {
                           ws[lay.W[i] + e] = x.w;
                           ws[lay.M[i] + e] = x.m;
                           if (a.save_states) { saved[(size_t)i * dh + e] = x.w; saved[(size_t)(NMAT + i) * dh + e] = x.m; }
                       });
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
        if (warp == kF64Warps - 1) chunk_scalars_warp<double>(eta + c * C, beta + c * C, gamma + c * C, min(C, L - c * C), &sh.sc[c & 1]);
    };
    tokens(0);
    scalars(0);
    if (tid == 0) {
        const double* W = ws + lay.W[0];
        const double* Wl = ws + lay.W[LAST];
        auto act = [&](F64Job& j, size_t x, size_t out) {
            f64_make(j, kEpiAct, h, -1 - C, NMAT - 1, 1, 1, h, sw);
            f64_seg(j, d, f64_op(W, d, 1), f64_op(ws + x, d, 1));
            if (sw) f64_a(j, 1, f64_op(ws + lay.W[1], d, 1));
            f64_out(j, 0, f64_ptr(ws + out));
        };
        for (int b = 0; b < 2; ++b) {  // by the chunk's parity
            F64Job& j = sh.job[b ? kFK1 : kFK];
            act(j, fl.fK[b], fl.fA);
            f64_out(j, 1, f64_ptr(ws + fl.fc1));
            if (sw) f64_out(j, 2, f64_ptr(ws + fl.fc2));
        }
        act(sh.job[kFQ], fl.fQ, fl.fAq);
        auto to_u = [&](F64Job& j, size_t x, size_t out) {
            f64_make(j, kEpiStore, d, -1 - C, 1, 1, 1, d, sw, parts);
            f64_seg(j, h, f64_op(Wl, h, 1), f64_op(ws + x, h, 1));
            f64_out(j, 0, f64_ptr(ws + out));
            j.pstride = (long long)pstride;
        };
        to_u(sh.job[kFU], fl.fA, fl.fUk);
        to_u(sh.job[kFUq], fl.fAq, fl.fUq);
        {
            F64Job& j = f64_make(sh.job[kFPz], kEpiPz, h, -1 - C, 1, 1, 1, h, sw);
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
                const int rows = i == LAST ? d : h, cols = i == LAST ? h : d;
                F64Job& j = f64_make(sh.job[(b ? kFUpd1 : kFUpd) + i], kEpiUpdate, rows, cols, 2, 0, cols, 1, sw);
                f64_seg(j, -1, f64_op(ws + (i == LAST ? fl.fPuW : fl.fPzW[i]), 1, rows), f64_op(ws + (i == LAST ? fl.fA : fl.fK[b]), 1, cols));
                f64_a(j, 1, f64_op(ws + (i == LAST ? fl.fPuM : fl.fPzM[i]), 1, rows));
                f64_inout(j, 0, f64_ptr(ws + lay.W[i]));
                f64_inout(j, 1, f64_ptr(ws + lay.M[i]));
                f64_out(j, 2, normed ? F64Ptr{nullptr, 0} : f64_ptr(saved + (size_t)i * dh));  // (normalised first: saved there)
                f64_out(j, 3, f64_ptr(saved + (size_t)(NMAT + i) * dh));
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
        const ChunkScalars<double>& sc = sh.sc[c & 1];
        cx.len = len;
        cx.kW = sc.kW; cx.kM = sc.kM; cx.cw = sc.cw; cx.cm = sc.cm; cx.cb = sc.cb;
        auto run = [&](int j0, int j1) { f64_jobs(sh.job, j0, j1, cx, rank, CL, f64_smem); };

        // Algorithm 1 line 1: the network, keys first
        const int odd = c & 1;
        run(kFK + odd, kFK + odd + 1);
        phase_sync(CL);
        run(kFU, a.o ? kFQ + 1 : kFQ);
        phase_sync(CL);
        // Algorithm 1 line 3: layer norm, e = f(k) - v and pu = dL/du for the key rows; tokens and scalars of the next chunk
        if (c + 1 < a.nchunks) {
            tokens(c + 1);
            scalars(c + 1);
        }
        for (int m = rank + CL * warp; m < len + (a.o && c > 0 ? C : 0); m += CL * kF64Warps) {
            if (m >= len) {  // rows of the queries of the chunk before
                output_row(c - 1, m - len);
                continue;
            }
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
                ws[fl.fPuM + (size_t)m * d + i] = x * sc.kM[m];
            }
        }
        phase_sync(CL);
        // back through the last matrix and the activation
        run(kFPz, a.o ? kFUq + 1 : kFUq);
        phase_sync(CL);
        // Algorithm 1 lines 4-7
        int slot = -1;  // the saved state that this chunk's end is
        if (a.save_states == 1 && (c + 1 < a.nchunks || normed)) slot = c + 1;
        else if (a.save_states == 2 && c + 1 < a.nchunks && (c + 1) % lay.seg == 0) slot = (c + 1) / lay.seg;
        cx.save = slot < 0 ? -1 : (long long)(slot * state_bytes);
        run(odd ? kFUpd1 : kFUpd, (odd ? kFUpd1 : kFUpd) + NMAT);
        phase_sync(CL);
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
    if (a.o)
        for (int m = rank + CL * warp; m < L - (a.nchunks - 1) * C; m += CL * kF64Warps) output_row(a.nchunks - 1, m);
    for (int i = 0; i < NMAT; ++i) {
        if (!a.W_final[i]) continue;  // recomputation for the reverse pass: only the saved states matter
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
    static std::atomic<int> state[64];
    constexpr size_t smem = kF64TileSmem + sizeof(F64FwdShared);
    static_assert(smem <= 232448, "227 KB of shared memory per CTA");
    return simt_launch(f64_fwd_kernel, a, kF64Threads, smem, state, reinterpret_cast<cudaStream_t>(stream), kind == 0 ? 0 : 1);
}

}  // namespace e2ttt
