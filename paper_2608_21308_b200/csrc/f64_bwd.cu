// Reverse pass for fp32 I/O in fp64: any d, h, C and both networks.  The adjoint of the chunk program, in matrix form over a chunk
// (notation: T, S = adjoints of the chunk-end (W, M); a trailing "b" marks an adjoint; "Wl" is the last matrix [d x h]):
//   GELU MLP : hidden a = gelu(z1)                 pz1 = ph gelu'(z1)
//   SwiGLU   : hidden a = silu(z1) z2              pz1 = ph z2 silu'(z1),  pz2 = ph silu(z1)
// Only what meets T and S is a chain over the chunks.  The chunks are taken in groups: f64_prepare_kernel re-runs each chunk's forward
// from the saved chunk-start state and reverses its outputs o = f_{W0}(q), all chunks of a group side by side on the whole GPU;
// f64_chain_kernel walks the group, five phases per chunk; f64_gate_kernel reverses the scans.  Products, tilings and what bounds them:
// f64_common.cuh.
#include "f64_common.cuh"

namespace e2ttt {

namespace {

struct F64GroupArgs {
    int N, cl;    // clusters and their CTAs
    int c0, ng;   // chunks of the group; chunk c0 + g has slot g
    int first, last;
    SimtBwdArgs a;
};

// second-order term of the activation needs no name of its own: se1 = ph f3, se2 = ph f4 (f64_act)
enum { kPK, kPQ, kPUk, kPUq, kPPz, kPZq, kPDq, kPJobs };
struct F64PrepareShared {
    F64Job job[kPJobs];
    ChunkScalars<double> sc;
};

__global__ void __launch_bounds__(kF64Threads, 1) f64_prepare_kernel(const F64GroupArgs ga, const int sw) {
    extern __shared__ __align__(16) unsigned char f64_smem[];
    F64PrepareShared& sh = *reinterpret_cast<F64PrepareShared*>(f64_smem + kF64TileSmem);
    const SimtBwdArgs& a = ga.a;
    const int CL = ga.cl, item = blockIdx.x / CL, rank = blockIdx.x % CL;
    const int seq = item / ga.ng, g = item % ga.ng, c = ga.c0 + g;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int NMAT = sw ? 3 : 2, LAST = NMAT - 1;
    const int d = a.d, h = a.h, C = a.C, s = c * C, len = min(C, a.L - s);
    const size_t dh = (size_t)d * h, tok = ((size_t)seq * a.Ls + s) * d;
    const F64Layout& fl = a.lay.fl;
    double* ws = reinterpret_cast<double*>(a.ws) + (size_t)seq * a.lay.per_seq;
    double* sl = ws + fl.slot + (size_t)g * fl.slot_stride;
    const float* kc = reinterpret_cast<const float*>(a.k) + tok;
    const float* qc = reinterpret_cast<const float*>(a.q) + tok;
    const float* vc = reinterpret_cast<const float*>(a.v) + tok;
    const float* doc = reinterpret_cast<const float*>(a.d_o) + tok;
    float* dqc = reinterpret_cast<float*>(a.dq) + tok;
    const int parts = f64_parts(C, d, h);
    const size_t pstride = (size_t)C * d;

    if (tid == 0) {
        const double* W = ws + a.lay.ckpt + (size_t)c * 2 * NMAT * dh;
        const double* Wl = W + (size_t)LAST * dh;
        auto act = [&](F64Job& j, size_t x) -> F64Job& {
            f64_make(j, kEpiAct, h, -1 - C, NMAT - 1, 1, 1, h, sw);
            f64_seg(j, d, f64_op(W, d, 1), f64_op(sl + x, d, 1));
            if (sw) f64_a(j, 1, f64_op(W + dh, d, 1));
            return j;
        };
        {
            F64Job& j = act(sh.job[kPK], fl.sK);
            f64_out(j, 0, f64_ptr(sl + fl.sAk));
            f64_out(j, 1, f64_ptr(sl + fl.sc1));
            f64_out(j, 3, f64_ptr(sl + fl.se1));
            if (sw) { f64_out(j, 2, f64_ptr(sl + fl.sc2)); f64_out(j, 4, f64_ptr(sl + fl.se2)); }
        }
        {
            F64Job& j = act(sh.job[kPQ], fl.sQ);
            f64_out(j, 0, f64_ptr(sl + fl.sAq));
            f64_out(j, 1, f64_ptr(sl + fl.szq[0]));
            if (sw) f64_out(j, 2, f64_ptr(sl + fl.szq[1]));
        }
        auto to_u = [&](F64Job& j, size_t x, size_t out) {
            f64_make(j, kEpiStore, d, -1 - C, 1, 1, 1, d, sw, parts);
            f64_seg(j, h, f64_op(Wl, h, 1), f64_op(sl + x, h, 1));
            f64_out(j, 0, f64_ptr(sl + out));
            j.pstride = (long long)pstride;
        };
        to_u(sh.job[kPUk], fl.sAk, fl.sUk);
        to_u(sh.job[kPUq], fl.sAq, fl.sUq);
        {
            F64Job& j = f64_make(sh.job[kPPz], kEpiPz, h, -1 - C, 1, 1, 1, h, sw);
            f64_seg(j, d, f64_op(Wl, 1, h), f64_op(sl + fl.sPu, d, 1));
            f64_pre(j, f64_ptr(sl + fl.sc1));
            f64_pre(j, f64_ptr(sl + (sw ? fl.sc2 : fl.se1)));
            if (sw) { f64_pre(j, f64_ptr(sl + fl.se1)); f64_pre(j, f64_ptr(sl + fl.se2)); }
            for (int i = 0; i < LAST; ++i) {
                f64_out(j, i, f64_ptr(sl + fl.sPz[i]));
                f64_out(j, 4 + 2 * i, f64_ptr(sl + fl.sPzW[i]));
                f64_out(j, 5 + 2 * i, f64_ptr(sl + fl.sPzM[i]));
                f64_out(j, LAST + i, f64_ptr(sl + (i ? fl.se2 : fl.se1)));
            }
        }
        {
            F64Job& j = f64_make(sh.job[kPZq], kEpiPz, h, -1 - C, 1, 1, 1, h, sw);
            f64_seg(j, d, f64_op(Wl, 1, h), f64_op(sl + fl.sUqb, d, 1));
            for (int i = 0; i < LAST; ++i) f64_inout(j, i, f64_ptr(sl + fl.szq[i]));
        }
        {
            F64Job& j = f64_make(sh.job[kPDq], kEpiDq, d, -1 - C, 1, 1, 1, d, sw);
            for (int i = 0; i < LAST; ++i) f64_seg(j, h, f64_op(W + (size_t)i * dh, 1, d), f64_op(sl + fl.szq[i], h, 1));
            j.ptr[kF64Aux] = f64_ptr(reinterpret_cast<double*>(const_cast<float*>(doc)));  // (floats)
            f64_out(j, 0, f64_ptr(reinterpret_cast<double*>(dqc)));
        }
    }
    for (int e = tid + rank * kF64Threads; e < len * d; e += kF64Threads * CL) {  // tokens -> fp64, for the products
        sl[fl.sK + e] = (double)kc[e];
        sl[fl.sQ + e] = (double)qc[e];
    }
    if (warp == kF64Warps - 1) {
        const size_t t0 = (size_t)seq * a.Ls + s;
        chunk_scalars_warp<double>(a.eta + t0, a.beta + t0, a.gamma + t0, len, &sh.sc);
        if (rank == 0) {  // what the chain needs of them
            double* o = sl + fl.ssc;
            __syncwarp();
            if (lane == 0) { o[0] = sh.sc.cw; o[1] = sh.sc.cm; o[2] = sh.sc.cb; }
            for (int t = lane; t < len; t += 32) { o[8 + t] = sh.sc.kW[t]; o[8 + C + t] = sh.sc.kM[t]; }
        }
    }
    __syncthreads();
    phase_sync(CL);
    F64Ctx cx{};
    cx.len = len;
    cx.kW = sh.sc.kW;
    cx.kM = sh.sc.kM;
    auto run = [&](int j0, int j1) { f64_jobs<kF64Bwd>(sh.job, j0, j1, cx, rank, CL, f64_smem); };
    auto u_row = [&](size_t up, int m, int i) { return f64_parts_at(sl + up, (size_t)m * d + i, parts, pstride); };
    const double inv = 1.0 / d;

    run(kPK, kPQ + 1);
    phase_sync(CL);
    run(kPUk, kPUq + 1);
    phase_sync(CL);
    // layer norm; e = f(k) - v and pu = dL/du for the key rows; adjoint of the outputs' layer norm
    for (int m = rank + CL * warp; m < 2 * len; m += CL * kF64Warps) {
        const bool key = m < len;
        const int t = key ? m : m - len;
        const size_t up = key ? fl.sUk : fl.sUq, row = (size_t)t * d;
        double* out = sl + (key ? fl.sPu : fl.sUqb) + row;
        double su = 0.0;
#pragma unroll 2
        for (int i = lane; i < d; i += 32) { const double x = u_row(up, t, i); out[i] = x; su += x; }
        const double mu = warp_sum(su) * inv;
        double var = 0.0;
#pragma unroll 2
        for (int i = lane; i < d; i += 32) { const double x = out[i] - mu; var += x * x; }
        const double r = r_rsqrt(warp_sum(var) * inv + (double)a.eps);
        auto e_of = [&](int i, double y) { return key ? (double)kc[row + i] + y - (double)vc[row + i] : (double)doc[row + i]; };
        double se = 0.0, sey = 0.0;
#pragma unroll 2
        for (int i = lane; i < d; i += 32) {
            const double y = (out[i] - mu) * r, e = e_of(i, y);
            se += e;
            sey += e * y;
        }
        se = warp_sum(se) * inv;
        sey = warp_sum(sey) * inv;
#pragma unroll 2
        for (int i = lane; i < d; i += 32) {
            const double y = (out[i] - mu) * r, x = r * (e_of(i, y) - se - y * sey);
            out[i] = x;
            if (key) {
                sl[fl.sY + row + i] = y;
                sl[fl.sPuW + row + i] = x * sh.sc.kW[t];
                sl[fl.sPuM + row + i] = x * sh.sc.kM[t];
            }
        }
        if (key && lane == 0) { sl[fl.sr + t] = r; sl[fl.smey + t] = sey; }
    }
    phase_sync(CL);
    run(kPPz, kPZq + 1);
    phase_sync(CL);
    run(kPDq, kPDq + 1);
}

enum { kCXY, kCX2, kCPub, kCKb, kCZ, kCDk, kCT, kCJobs = kCT + 3 };
struct F64ChainShared {
    F64Job job[kCJobs];
    double kW[kMaxC], kM[kMaxC];
};

__global__ void __launch_bounds__(kF64Threads, 1) f64_chain_kernel(const F64GroupArgs ga, const int sw) {
    extern __shared__ __align__(16) unsigned char f64_smem[];
    F64ChainShared& sh = *reinterpret_cast<F64ChainShared*>(f64_smem + kF64TileSmem);
    const SimtBwdArgs& a = ga.a;
    const int CL = ga.cl, seq = blockIdx.x / CL, rank = blockIdx.x % CL;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int NMAT = sw ? 3 : 2, LAST = NMAT - 1;
    const int d = a.d, h = a.h, C = a.C;
    const size_t dh = (size_t)d * h;
    const SimtLayout& lay = a.lay;
    const F64Layout& fl = lay.fl;
    double* ws = reinterpret_cast<double*>(a.ws) + (size_t)seq * lay.per_seq;
    float* dk = reinterpret_cast<float*>(a.dk) + (size_t)seq * a.Ls * d;
    float* dv = reinterpret_cast<float*>(a.dv) + (size_t)seq * a.Ls * d;
    const int parts = f64_parts(C, d, h);
    const size_t pstride = (size_t)C * d;
    const int c1 = ga.c0 + ga.ng - 1;  // the first chunk
    const long long scs = -(long long)(fl.slot_stride * sizeof(double)), ccs = -(long long)(2 * NMAT * dh * sizeof(double));
    auto slot_of = [&](int c) { return ws + fl.slot + (size_t)(c - ga.c0) * fl.slot_stride; };

    if (ga.first && !a.carry_in)
        for (int i = 0; i < NMAT; ++i) {
            const float* tf = a.dW_final[i] ? a.dW_final[i] + (size_t)seq * dh : nullptr;
            const float* sf = a.dM_final[i] ? a.dM_final[i] + (size_t)seq * dh : nullptr;
            struct TS { double t, s; };
            batched_for<8>(tid + (size_t)rank * kF64Threads, dh, (size_t)kF64Threads * CL,
                           [&](size_t e) { return TS{tf ? (double)tf[e] : 0.0, sf ? (double)sf[e] : 0.0}; },
                           [&](size_t e, const TS& x) { ws[lay.T[i] + e] = x.t; ws[lay.S[i] + e] = x.s; });
        }
    if (tid == 0) {
        double* s0 = slot_of(c1);
        auto slot_op = [&](size_t off, int rs, int ks) { return f64_op(s0 + off, rs, ks, scs); };
        auto slot_ptr = [&](size_t off) { return f64_ptr(s0 + off, scs); };
        double* ck = ws + lay.ckpt + (size_t)c1 * 2 * NMAT * dh;
        auto W_op = [&](int i, int rs, int ks) { return f64_op(ck + (size_t)i * dh, rs, ks, ccs); };
        auto T = [&](int i) { return ws + lay.T[i]; };
        auto S = [&](int i) { return ws + lay.S[i]; };
        {  // x = T k, y = S k of the first matrices: adjoint of pz; through it to phb, the first part of zb, shares of those of K^W, K^M
            F64Job& j = f64_make(sh.job[kCXY], kEpiXY, h, -1 - C, 2 * LAST, 1, 1, h, sw);
            f64_seg(j, d, f64_op(T(0), d, 1), slot_op(fl.sK, d, 1));
            f64_a(j, 1, f64_op(S(0), d, 1));
            if (sw) { f64_a(j, 2, f64_op(T(1), d, 1)); f64_a(j, 3, f64_op(S(1), d, 1)); }
            for (int i = 0; i < LAST; ++i) {
                f64_pre(j, slot_ptr(fl.sPz[i]));
                f64_pre(j, slot_ptr(i ? fl.sc2 : fl.sc1));
                f64_pre(j, slot_ptr(i ? fl.se2 : fl.se1));
                f64_out(j, 1 + i, f64_ptr(ws + fl.zb[i]));
            }
            f64_out(j, 0, f64_ptr(ws + fl.phb));
            j.ptr[kF64Aux] = f64_ptr(ws + fl.kwp);
            j.auxn = C;
        }
        auto tok_d = [&](F64Job& j, int na, size_t out) -> F64Job& {  // a [tokens x d] result in parts
            f64_make(j, kEpiStore, d, -1 - C, na, 1, 1, d, sw, parts);
            f64_out(j, 0, f64_ptr(ws + out));
            j.pstride = (long long)pstride;
            return j;
        };
        {
            F64Job& j = tok_d(sh.job[kCX2], 2, fl.X2);
            f64_seg(j, h, f64_op(T(LAST), h, 1), slot_op(fl.sAk, h, 1));
            f64_a(j, 1, f64_op(S(LAST), h, 1));
            f64_out(j, 1, f64_ptr(ws + fl.Y2));
        }
        f64_seg(tok_d(sh.job[kCPub], 1, fl.Pub), h, W_op(LAST, h, 1), f64_op(ws + fl.phb, h, 1));
        {  // minus this is a part of dk
            F64Job& j = tok_d(sh.job[kCKb], 1, fl.Kb);
            for (int i = 0; i < LAST; ++i) {
                f64_seg(j, h, f64_op(T(i), 1, d), slot_op(fl.sPzW[i], h, 1));
                f64_seg(j, h, f64_op(S(i), 1, d), slot_op(fl.sPzM[i], h, 1));
            }
        }
        {  // minus the adjoint of the hidden activation -> zb
            F64Job& j = f64_make(sh.job[kCZ], kEpiZ, h, -1 - C, 1, 1, 1, h, sw);
            f64_seg(j, d, f64_op(T(LAST), 1, h), slot_op(fl.sPuW, d, 1));
            f64_seg(j, d, f64_op(S(LAST), 1, h), slot_op(fl.sPuM, d, 1));
            f64_seg(j, d, W_op(LAST, 1, h), f64_op(ws + fl.nUkb, d, 1));
            for (int i = 0; i < LAST; ++i) {
                f64_inout(j, i, f64_ptr(ws + fl.zb[i]));
                f64_pre(j, slot_ptr(i ? fl.sc2 : fl.sc1));
            }
        }
        {
            F64Job& j = tok_d(sh.job[kCDk], 1, fl.dk);
            for (int i = 0; i < LAST; ++i) f64_seg(j, h, W_op(i, 1, d), f64_op(ws + fl.zb[i], h, 1));
        }
        const size_t dots = (size_t)f64_tiles(h, d, f64_wide(h, d) ? 32 : 16) * kF64Warps * 3;
        for (int i = 0; i < NMAT; ++i) {
            F64Job& j = f64_make(sh.job[kCT + i], kEpiT, i == LAST ? d : h, i == LAST ? h : d, 1, 0, i == LAST ? h : d, 1, sw);
            if (i < LAST) {
                f64_seg(j, -1, slot_op(fl.szq[i], 1, h), slot_op(fl.sQ, 1, d));
                f64_seg(j, -1, f64_op(ws + fl.zb[i], 1, h), slot_op(fl.sK, 1, d));
            } else {
                f64_seg(j, -1, slot_op(fl.sUqb, 1, d), slot_op(fl.sAq, 1, h));
                f64_seg(j, -1, slot_op(fl.sPu, 1, d), f64_op(ws + fl.phb, 1, h));
                f64_seg(j, -1, f64_op(ws + fl.Ukb, 1, d), slot_op(fl.sAk, 1, h));
            }
            f64_inout(j, 0, f64_ptr(T(i)));
            f64_inout(j, 1, f64_ptr(S(i)));
            f64_pre(j, f64_ptr(ck + (size_t)i * dh, ccs));
            f64_pre(j, f64_ptr(ck + (size_t)(NMAT + i) * dh, ccs));
            j.ptr[kF64Aux] = slot_ptr(fl.sdots + i * dots);
        }
    }
    __syncthreads();
    phase_sync(CL);

    const double inv = 1.0 / d;
    F64Ctx cx{};
    cx.kW = sh.kW;
    cx.kM = sh.kM;
    auto run = [&](int j0, int j1) { f64_jobs<kF64Bwd>(sh.job, j0, j1, cx, rank, CL, f64_smem); };
    auto dk_rows = [&](int c) {
        const int s = c * C, len = min(C, a.L - s);
        for (int t = rank + CL * warp; t < len; t += CL * kF64Warps)
#pragma unroll 2
            for (int i = lane; i < d; i += 32) {
                const size_t e = (size_t)t * d + i;
                dk[(size_t)s * d + e] = (float)(ws[fl.Eb + e] - f64_parts_at(ws + fl.Kb, e, parts, pstride) + f64_parts_at(ws + fl.dk, e, parts, pstride));
            }
    };
    for (int c = c1; c >= ga.c0; --c) {
        const int s = c * C, len = min(C, a.L - s);
        double* sl = slot_of(c);
        cx.len = len;
        const double* scal = sl + fl.ssc;
        for (int t = tid; t < len; t += kF64Threads) { sh.kW[t] = scal[8 + t]; sh.kM[t] = scal[8 + C + t]; }
        cx.cw = scal[0]; cx.cm = scal[1]; cx.cb = scal[2];

        // post-chunk normalisation (optional): T arrives as the adjoint of the normalised chunk-end weights
        // y = n w / (s + eps_n), s = ||w||.  With y itself (the next chunk's saved start state) and the saved s:
        //   w_bar = n/(s + eps_n) y_bar - y <y_bar, y> / (n s),      n_bar = <y_bar, y> / n
        if (a.row_norm[0]) {
            const int maxdim = d > h ? d : h;
            const double* nxt = ws + lay.ckpt + (size_t)(c + 1) * 2 * NMAT * dh;
            for (int i = 0; i < NMAT; ++i) {
                const int rows = (i == LAST) ? d : h, cols = (i == LAST) ? h : d;
                const float* target = a.row_norm[i] + (size_t)seq * rows;
                float* tb = a.d_row_norm[i] ? a.d_row_norm[i] + (size_t)seq * rows : nullptr;
                for (int r = warp + rank * kF64Warps; r < rows; r += kF64Warps * CL) {
                    double* t = ws + lay.T[i] + (size_t)r * cols;
                    const double* y = nxt + (size_t)i * dh + (size_t)r * cols;
                    double ty = 0.0;
#pragma unroll 2
                    for (int j = lane; j < cols; j += 32) ty += t[j] * y[j];
                    ty = warp_sum(ty);
                    const double n = (double)target[r], nrm = ws[lay.rown + ((size_t)c * 3 + i) * maxdim + r];
                    const double f = n / (nrm + (double)a.norm_eps);
                    const double g = (n != 0.0 && nrm > 0.0) ? ty / (n * nrm) : 0.0;
#pragma unroll 2
                    for (int j = lane; j < cols; j += 32) t[j] = f * t[j] - y[j] * g;
                    if (tb && lane == 0) {
                        const double nb = (n != 0.0) ? ty / n : 0.0;
                        tb[r] = (c == a.nchunks - 1) ? (float)nb : tb[r] + (float)nb;
                    }
                }
            }
            phase_sync(CL);
        }

        // ---- everything that meets T, S first; dk of the chunk before
        if (c < c1) dk_rows(c + 1);
        run(kCXY, kCX2 + 1);
        phase_sync(CL);
        run(kCPub, kCKb + 1);
        phase_sync(CL);
        // ---- rows: pu = J(u) e, e = k + y - v, y = LN(u): adjoints of e and u; dv; adjoints of K^W, K^M
        {
            const int ntm = (h + (sh.job[kCXY].wide ? 31 : 15)) / (sh.job[kCXY].wide ? 32 : 16);
            for (int t = rank + CL * warp; t < len; t += CL * kF64Warps) {
                const size_t row = (size_t)t * d;
                const double *y = sl + fl.sY + row, *pu = sl + fl.sPu + row;
                double *eb = ws + fl.Eb + row, *ub = ws + fl.Ukb + row;
                const double r = sl[fl.sr + t], mey = sl[fl.smey + t], kw = sh.kW[t], km = sh.kM[t];
                double wb = 0.0, mb = 0.0, sx = 0.0, mpy = 0.0, spp = 0.0;
#pragma unroll 2
                for (int j = lane; j < ntm; j += 32) {
                    wb += ws[fl.kwp + (size_t)j * C + t];
                    mb += ws[fl.kwp + (size_t)(ntm + j) * C + t];
                }
#pragma unroll 2
                for (int i = lane; i < d; i += 32) {
                    const double x = f64_parts_at(ws + fl.X2, row + i, parts, pstride), x2 = f64_parts_at(ws + fl.Y2, row + i, parts, pstride);
                    const double p = pu[i], pub = f64_parts_at(ws + fl.Pub, row + i, parts, pstride) - (kw * x + km * x2);
                    wb += p * x;
                    mb += p * x2;
                    sx += pub;
                    mpy += pub * y[i];
                    spp += pub * p;
                    eb[i] = pub;
                }
                wb = warp_sum(wb); mb = warp_sum(mb);
                if (lane == 0) { sl[fl.skwb + t] = -wb; sl[fl.skwb + C + t] = -mb; }
                sx = warp_sum(sx) * inv; mpy = warp_sum(mpy) * inv; spp = warp_sum(spp);
                double s2 = 0.0, s2y = 0.0;
#pragma unroll 2
                for (int i = lane; i < d; i += 32) {
                    const double e = r * (eb[i] - sx - y[i] * mpy);
                    eb[i] = e;
                    s2 += e;
                    s2y += e * y[i];
                    dv[(size_t)s * d + row + i] = (float)-e;
                }
                s2 = warp_sum(s2) * inv; s2y = warp_sum(s2y) * inv;
                // second-order term of the LN Jacobian, and dy -> du for the y inside e
#pragma unroll 2
                for (int i = lane; i < d; i += 32) {
                    const double x = r * (eb[i] - s2 - y[i] * s2y) - r * inv * spp * y[i] - r * (mpy * pu[i] + mey * eb[i]);
                    ub[i] = x;
                    ws[fl.nUkb + row + i] = -x;
                }
            }
        }
        phase_sync(CL);
        run(kCZ, kCZ + 1);
        phase_sync(CL);
        // ---- dk = .. + zb W; adjoints of the chunk-start state, and of the carries
        run(kCDk, kCT + NMAT);
        f64_step(sh.job, kCT + NMAT);
        phase_sync(CL);
    }
    dk_rows(ga.c0);
    if (ga.last && !a.carry_out)
        for (int i = 0; i < NMAT; ++i) {
            float* wf = a.dW_init[i] + (size_t)seq * dh;
            float* mf = a.dM_init[i] + (size_t)seq * dh;
            struct TS { double t, s; };
            batched_for<8>(tid + (size_t)rank * kF64Threads, dh, (size_t)kF64Threads * CL,
                           [&](size_t e) { return TS{ws[lay.T[i] + e], ws[lay.S[i] + e]}; },
                           [&](size_t e, const TS& x) { wf[e] = (float)x.t; mf[e] = (float)x.s; });
        }
}

// Reverse of the suffix scans: one CTA per chunk.  One thread walks the chunk (a 3-term linear recurrence, ~10 flop per token); its
// operands are brought into shared memory first and its results leave the same way, so the walk itself never waits for global memory.
struct F64GateShared {
    ChunkScalars<double> sc;
    double red[3][kF64Warps];
    double beta[kMaxC], gamma[kMaxC], eta[kMaxC], kWb[kMaxC], kMb[kMaxC], de[kMaxC], db[kMaxC], dg[kMaxC];
};
__global__ void __launch_bounds__(kF64Threads, 1) f64_gate_kernel(const F64GroupArgs ga, const int sw) {
    extern __shared__ __align__(16) unsigned char f64_smem[];
    F64GateShared& sh = *reinterpret_cast<F64GateShared*>(f64_smem);
    const SimtBwdArgs& a = ga.a;
    const int seq = blockIdx.x / ga.ng, g = blockIdx.x % ga.ng, c = ga.c0 + g;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int C = a.C, s = c * C, len = min(C, a.L - s);
    const F64Layout& fl = a.lay.fl;
    const double* sl = reinterpret_cast<const double*>(a.ws) + (size_t)seq * a.lay.per_seq + fl.slot + (size_t)g * fl.slot_stride;
    const size_t t0 = (size_t)seq * a.Ls + s;
    // adjoints of the carries: shares of tiles and warps, in a fixed order
    {
        const int n = (sw ? 3 : 2) * f64_tiles(a.h, a.d, f64_wide(a.h, a.d) ? 32 : 16) * kF64Warps;
        double x[3] = {0.0, 0.0, 0.0};
        for (int i = tid; i < n; i += kF64Threads)
#pragma unroll
            for (int j = 0; j < 3; ++j) x[j] += sl[fl.sdots + (size_t)i * 3 + j];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            x[j] = warp_sum(x[j]);
            if (lane == 0) sh.red[j][warp] = x[j];
        }
    }
    if (warp == 0) chunk_scalars_warp<double>(a.eta + t0, a.beta + t0, a.gamma + t0, len, &sh.sc);
    for (int t = tid; t < len; t += kF64Threads) {
        sh.beta[t] = (double)a.beta[t0 + t];
        sh.gamma[t] = (double)a.gamma[t0 + t];
        sh.eta[t] = (double)a.eta[t0 + t];
        sh.kWb[t] = sl[fl.skwb + t];
        sh.kMb[t] = sl[fl.skwb + C + t];
    }
    __syncthreads();
    if (tid == 0) {
        double cb[3] = {0.0, 0.0, 0.0};  // adjoints of cw, cm, cb
        for (int j = 0; j < 3; ++j)
            for (int w = 0; w < kF64Warps; ++w) cb[j] += sh.red[j][w];
        double Sb = 0.0, btb = cb[2], gtb = cb[0];  // adjoints of S_0 (unused), bt_0, gt_0
        for (int t = 0; t < len; ++t) {  // index t: state t; token t+1 lives at array index t
            const double b1 = sh.beta[t], g1 = sh.gamma[t], e1 = sh.eta[t], kWb = sh.kWb[t], kMb = sh.kMb[t];
            const double S1 = sh.sc.S[t + 1], bt1 = sh.sc.bt[t + 1];
            // S_t = beta_{t+1} S_{t+1} + gt_t ; bt_t = beta_{t+1} bt_{t+1} ; gt_t = gamma_{t+1} gt_{t+1}
            gtb += Sb;
            double bb = Sb * S1 + btb * bt1, Sn = Sb * b1;
            const double gb = gtb * sh.sc.gt[t + 1];
            if (t == 0) {  // cm = beta_1 S_1
                bb += cb[1] * S1;
                Sn += cb[1] * b1;
            }
            // K^M_{t+1} = eta bt_{t+1}, K^W_{t+1} = eta S_{t+1}
            sh.de[t] = kMb * bt1 + kWb * S1;
            sh.db[t] = bb;
            sh.dg[t] = gb;
            Sb = Sn + kWb * e1;
            btb = btb * b1 + kMb * e1;
            gtb = gtb * g1;
        }
    }
    __syncthreads();
    for (int t = tid; t < len; t += kF64Threads) {
        a.d_eta[t0 + t] = (float)sh.de[t];
        a.d_beta[t0 + t] = (float)sh.db[t];
        a.d_gamma[t0 + t] = (float)sh.dg[t];
    }
}

}  // namespace

int f64_bwd_launch(const SimtBwdArgs& a, int kind, void* stream) {
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    static std::atomic<int> state[3][64];
    constexpr size_t prepare_smem = kF64TileSmem + sizeof(F64PrepareShared), chain_smem = kF64TileSmem + sizeof(F64ChainShared);
    static_assert(prepare_smem <= 232448 && chain_smem <= 232448 && sizeof(F64GateShared) <= 232448, "227 KB of shared memory per CTA");
    const int sw = kind == 0 ? 0 : 1, G = a.lay.fl.G;
    for (int end = a.nchunks; end > 0;) {
        F64GroupArgs ga{};
        ga.a = a;
        ga.ng = G < end ? G : end;
        ga.c0 = end - ga.ng;
        ga.first = end == a.nchunks;
        ga.last = ga.c0 == 0;
        // a cluster per chunk and sequence, as large as one wave allows
        ga.N = a.N * ga.ng;
        ga.cl = simt_cluster_size(ga.N, 1);
        int rc = simt_launch(f64_prepare_kernel, ga, kF64Threads, prepare_smem, prepare_smem, state[0], st, sw);
        if (rc) return rc;
        ga.N = a.N;
        ga.cl = a.cl;
        rc = simt_launch(f64_chain_kernel, ga, kF64Threads, chain_smem, chain_smem, state[1], st, sw);
        if (rc) return rc;
        ga.N = a.N * ga.ng;
        ga.cl = 1;
        rc = simt_launch(f64_gate_kernel, ga, kF64Threads, sizeof(F64GateShared), sizeof(F64GateShared), state[2], st, sw);
        if (rc) return rc;
        end = ga.c0;
    }
    return 0;
}

}  // namespace e2ttt
