// Reverse pass on the block-tiled engine (tile.cuh): the adjoint of the chunk program for bf16 I/O, d <= 128, any h and C, both
// networks.  The mathematics is simt_bwd.cu's; this is another division of the work.
//
// Only what depends on the adjoints (T, S) of the chunk-end state forms a chain over the chunks.  Everything else - the
// chunk's forward, the adjoint of the outputs, the gradient with respect to q - is a function of the saved chunk-start state and the
// tokens alone.  So the chunks are taken in groups of G, from the last to the first, with four launches per group:
//   tile_prep   chunk-start weights and tokens -> operand blocks; scalar kernels of every chunk              (any order; inside
//               tile_rec for chunks of up to 64 tokens)
//   tile_rec    per (sequence, chunk, 64 tokens): forward of the chunk, pu, pz, adjoint of the outputs, dq   (any order)
//   tile_rev    per sequence: the chain over the group's chunks; a cluster of CTAs splits the hidden units
//   tile_gate   per (sequence, chunk): reverse of the suffix scans -> gate gradients                        (any order)
// With few sequences the chain leaves SMs idle: its launch then takes the next group's tile_rec along (two sets of slots).
// Notation: T, S = adjoints of (W, M) at the chunk end; a trailing "b" marks an adjoint; the first matrices are [h x d], the
// last one [d x h].
#include "simt_layout.h"
#include "tile_rec.cuh"

namespace e2ttt {
using namespace tile;

namespace {

// ---- operand blocks of the chunk-start weights and of the tokens; scalar kernels --------------------------------------------
template <int NMAT> __global__ void __launch_bounds__(256) tile_prep_kernel(const GroupArgs ga) {
    const int seq = blockIdx.x / ga.ng, g = blockIdx.x % ga.ng;
    prepare_chunk<NMAT>(ga.a, seq, ga.c0 + g, slot_of(ga.a, seq, ga.s0 + g), blockIdx.y * 8 + (threadIdx.x >> 5), gridDim.y * 8, threadIdx.x & 31);
}

template <int KIND> __global__ void __launch_bounds__(kThreads, 1) tile_rec_kernel(const GroupArgs ga) {
    extern __shared__ unsigned char tile_smem[];
    rec_items<KIND>(ga.a, NextGroup{ga.c0, ga.ng, ga.s0}, tile_smem, blockIdx.x, gridDim.x);
}

// ---- the chain over the chunks ---------------------------------------------------------------------------------------------------
struct RevShared {
    float kw[kMaxC], km[kMaxC];
    float red[kMaxC / 64][4][64][2];  // per token: the lane quadrants' shares of the adjoints of K^W_t, K^M_t
    float dots[kEpiWarps][4];
};

template <int KIND> __global__ void __launch_bounds__(kThreads, 1) tile_rev_kernel(const GroupArgs ga) {
    constexpr int NMAT = (KIND == 0) ? 2 : 3, LAST = NMAT - 1;
    constexpr bool SW = KIND == 1;
    extern __shared__ unsigned char tile_smem[];
    unsigned char* ring = tile_smem + ((1024u - (smem_u32(tile_smem) & 1023u)) & 1023u);
    Sync* sy = reinterpret_cast<Sync*>(ring + kUnits * kUnitBytes);
    RevShared& sh = *reinterpret_cast<RevShared*>(sy + 1);
    const SimtBwdArgs& a = ga.a;
    const int CL = a.cl, seq = blockIdx.x / CL, rank = blockIdx.x % CL;
    Engine G;
    G.setup(ring, sy, a.status, rank, CL);
    const int warp = G.warp, lane = G.lane, q4 = warp & 3, grp = warp >> 2, row = 32 * q4 + lane;
    const SimtLayout& lay = a.lay;
    const TileLayout& tl = lay.tl;
    const int d = a.d, h = a.h, db = tl.db, hb = tl.hb, tb = tl.tb, dp = db * 64;
    const size_t dh = (size_t)d * h;
    const int sb = (hb + CL - 1) / CL, hb0 = min(hb, rank * sb), hb1 = min(hb, hb0 + sb), nsl = hb1 - hb0;
    float* ws = reinterpret_cast<float*>(a.ws) + (size_t)seq * lay.per_seq;
    auto blk = [&](size_t off) { return bytes_of(ws + off); };
    const bool normed = a.row_norm[0] != nullptr;

    // operand blocks of a master of the chain, own hidden units
    auto to_blocks = [&](int i, const float* src, size_t dst) {
        if (i < LAST) matrix_to_blocks(src, d, h, 0, db, hb0, hb1, blk(dst), 1, db, warp, kEpiWarps, lane);
        else matrix_to_blocks(src, h, d, hb0, hb1, 0, db, blk(dst), db, 1, warp, kEpiWarps, lane);
    };
    if (ga.first && !a.carry_in) {
        if (G.epi()) {
#pragma unroll
            for (int i = 0; i < NMAT; ++i) {
                const float* tf = a.dW_final[i] ? a.dW_final[i] + (size_t)seq * dh : nullptr;
                const float* sf = a.dM_final[i] ? a.dM_final[i] + (size_t)seq * dh : nullptr;
                float *T = ws + lay.T[i], *S = ws + lay.S[i];
                batched_for<8>(threadIdx.x + (size_t)rank * kEpiThreads, dh, (size_t)kEpiThreads * CL,
                               [&](size_t e) { return make_float2(tf ? tf[e] : 0.0f, sf ? sf[e] : 0.0f); },
                               [&](size_t e, const float2& x) { T[e] = x.x; S[e] = x.y; });
            }
        }
        G.sync_cluster();
        if (G.epi()) {
#pragma unroll
            for (int i = 0; i < NMAT; ++i) {
                to_blocks(i, ws + lay.T[i], tl.Tb[i]);
                to_blocks(i, ws + lay.S[i], tl.Sb[i]);
            }
        }
        G.sync_cta();
    }

    // dk of a chunk = its e-adjoint + the CTAs' partial sums, in CTA order; rows dealt to the cluster's warps
    auto finish_dk = [&](int c, int buf) {
        const int s = c * a.C, len = min(a.C, a.L - s), ci = 4 * lane;
        __nv_bfloat16* dkc = reinterpret_cast<__nv_bfloat16*>(a.dk) + ((size_t)seq * a.Ls + s) * d;
        for (int t = rank * kEpiWarps + warp; t < len; t += CL * kEpiWarps) {
            if (ci >= dp) continue;
            const float4 x = *reinterpret_cast<const float4*>(ws + tl.bEb[buf] + (size_t)t * dp + ci);
            float o[4] = {x.x, x.y, x.z, x.w};
            add_parts(ws + tl.bdk[buf] + (size_t)t * dp + ci, 2 * CL, (size_t)tb * 64 * dp, o);
            st_tok4(dkc + (size_t)t * d, ci, d, o);
        }
    };

    for (int g = ga.ng - 1; g >= 0; --g) {
        const int c = ga.c0 + g, s = c * a.C, len = min(a.C, a.L - s), tbn = (len + 63) / 64, buf = c & 1;
        float* sl = slot_of(a, seq, ga.s0 + g);
        auto sblk = [&](size_t off) { return bytes_of(sl + off); };
        const ChunkScalars<float>& sc = *reinterpret_cast<const ChunkScalars<float>*>(sl + tl.ssc);
        const float* ck = ws + lay.ckpt + (size_t)c * 2 * NMAT * dh;
        for (int t = threadIdx.x; t < tbn * 64; t += kThreads) {
            sh.kw[t] = t < len ? sc.kW[t] : 0.0f;
            sh.km[t] = t < len ? sc.kM[t] : 0.0f;
        }

        if (normed) {
            // T arrives as the adjoint of the normalised chunk-end weights y = n w / (||w|| + eps_n); with y itself (the next
            // chunk's saved start state) and the saved norm:  w_bar = n/(s + eps_n) y_bar - y <y_bar, y> / (n s),  n_bar = <y_bar, y> / n
            G.sync_cluster();  // the previous chunk's T is complete
            if (G.epi()) {
                const int maxdim = d > h ? d : h;
                const float* nxt = ck + (size_t)2 * NMAT * dh;
#pragma unroll
                for (int i = 0; i < NMAT; ++i) {
                    const int rows = (i == LAST) ? d : h, cols = (i == LAST) ? h : d;
                    const float* target = a.row_norm[i] + (size_t)seq * rows;
                    float* tbar = a.d_row_norm[i] ? a.d_row_norm[i] + (size_t)seq * rows : nullptr;
                    for (int r = rank * kEpiWarps + warp; r < rows; r += CL * kEpiWarps) {
                        float* t = ws + lay.T[i] + (size_t)r * cols;
                        const float* y = nxt + (size_t)i * dh + (size_t)r * cols;
                        float ty = 0.0f;
                        for (int j = lane; j < cols; j += 32) ty += t[j] * y[j];
                        ty = warp_sum(ty);
                        const float n = target[r], nrm = ws[lay.rown + ((size_t)c * 3 + i) * maxdim + r];
                        const float f = n / (nrm + a.norm_eps), gy = (n != 0.0f && nrm > 0.0f) ? ty / (n * nrm) : 0.0f;
                        for (int j = lane; j < cols; j += 32) t[j] = f * t[j] - y[j] * gy;
                        if (tbar && lane == 0) {
                            const float nb = n != 0.0f ? ty / n : 0.0f;
                            tbar[r] = (c == a.nchunks - 1) ? nb : tbar[r] + nb;
                        }
                    }
                }
            }
            G.sync_cluster();
            if (G.epi())
#pragma unroll
                for (int i = 0; i < NMAT; ++i) to_blocks(i, ws + lay.T[i], tl.Tb[i]);
            G.sync_cta();
        } else {
            __syncthreads();
        }

        // A hidden-unit tile of a matrix as the lane-side operand with contraction over d: blocks (h, d), rows = d for the first
        // matrices (MN-major), rows = h for the last (K-major)
        auto by_h = [&](const unsigned char* m, int b0, bool two, bool first) {
            const unsigned char* p = m + (size_t)b0 * db * B;
            return Opnd{p, two ? p + (size_t)db * B : nullptr, B, true, first};
        };
        // the matrix with d on the lanes and contraction over the CTA's hidden units
        auto by_d = [&](const unsigned char* m, bool first) {
            const unsigned char* p = m + (size_t)hb0 * db * B;
            return Opnd{p, db == 2 ? p + B : nullptr, (uint32_t)db * B, true, !first};
        };
        // [h x tokens] blocks of 64 tokens as the column-side operand, contraction over the CTA's hidden units
        auto tok_h = [&](const unsigned char* m, int tk) {
            return Opnd{m + ((size_t)hb0 * tb + tk) * B, nullptr, (uint32_t)tb * B, true, true};
        };
        auto partial = [&](size_t base, int part, int tk) { return ws + base + ((size_t)(rank * 2 + part) * tb * 64 + tk * 64) * dp; };

        // ---- everything that meets (T, S) directly.  G_t enters W_C with K^W_t and M_C with K^M_t: its adjoint is K^W_t T + K^M_t S
        for (int tk = 0; tk < tbn; ++tk) {
            float kwb = 0.0f, kmb = 0.0f;  // of token 16 grp + (lane >> 1), this warp's hidden units
            for (int b0 = hb0; b0 < hb1; b0 += 2) {
                const bool two = b0 + 1 < hb1;
                // x = T_first k, y = S_first k: adjoint of pz; through pz = ph act'(z) to phb and the second-order part of zb
                {
                    const Opnd kt{sblk(tl.sK) + (size_t)tk * db * kHalf, nullptr, kHalf, false, false};
                    G.job_begin();
                    if constexpr (SW) {
                        const Opnd p[4] = {by_h(blk(tl.Tb[0]), b0, two, true), by_h(blk(tl.Sb[0]), b0, two, true),
                                           by_h(blk(tl.Tb[1]), b0, two, true), by_h(blk(tl.Sb[1]), b0, two, true)};
                        G.term<4>(db, false, kt, p, {0u, 64u, 128u, 192u});
                    } else {
                        const Opnd p[2] = {by_h(blk(tl.Tb[0]), b0, two, true), by_h(blk(tl.Sb[0]), b0, two, true)};
                        G.term<2>(db, false, kt, p, {0u, 64u});
                    }
                    G.job_end([&](uint32_t t) {
                        const int bl = b0 + (row >> 6), tok = 16 * grp;
                        const bool ok = row < 64 || two;
                        const size_t e0 = ok ? (((size_t)bl * tb + tk) * 64 + tok) * 64 + (row & 63) : 0;
                        const float* kw = sh.kw + tk * 64 + tok;
                        const float* km = sh.km + tk * 64 + tok;
                        float x[16], y[16], phb[16], z0[16], ph[16], cv[16];
                        auto ld_col = [&](size_t src, float (&v)[16]) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) v[j] = ok ? sl[src + e0 + 64 * j] : 0.0f;
                        };
                        ld_col(tl.sph, ph);
                        ld_col(tl.sc1, cv);
                        ld_col(tl.sc4, z0);
                        acc16(t + tok, x);
                        acc16(t + 64 + tok, y);
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const float pz = ph[j] * cv[j], pzb = -(kw[j] * x[j] + km[j] * y[j]);
                            x[j] = ok ? x[j] * pz : 0.0f;
                            y[j] = ok ? y[j] * pz : 0.0f;
                            phb[j] = pzb * cv[j];
                            z0[j] *= pzb;
                            if (SW) cv[j] = pzb;
                        }
                        kwb -= reduce16(x, lane);
                        kmb -= reduce16(y, lane);
                        if (SW) {
                            ld_col(tl.sg1, x);
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                x[j] *= ph[j];  // ph silu'(z1)
                                if (ok) ws[tl.bz0[LAST - 1] + e0 + 64 * j] = cv[j] * x[j];
                            }
                            ld_col(tl.sc2, cv);
                            float x2[16];
                            acc16(t + 128 + tok, x2);
                            acc16(t + 192 + tok, y);
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                const float pz = ph[j] * cv[j], pzb = -(kw[j] * x2[j] + km[j] * y[j]);
                                x2[j] = ok ? x2[j] * pz : 0.0f;
                                y[j] = ok ? y[j] * pz : 0.0f;
                                phb[j] += pzb * cv[j];
                                z0[j] += pzb * x[j];
                            }
                            kwb -= reduce16(x2, lane);
                            kmb -= reduce16(y, lane);
                        }
                        if (ok)
#pragma unroll
                            for (int j = 0; j < 16; ++j) ws[tl.bz0[0] + e0 + 64 * j] = z0[j];
                        if (ok) st_split16(blk(tl.bPhb) + ((size_t)bl * tb + tk) * B, row & 63, tok, phb);
                    });
                }
                // T_last^T pu, S_last^T pu: adjoint of the activation through the aggregation of the last matrix
                {
                    const Opnd pu{sblk(tl.sPu) + (size_t)tk * db * B, nullptr, B, true, false};
                    const Opnd p[2] = {by_h(blk(tl.Tb[LAST]), b0, two, false), by_h(blk(tl.Sb[LAST]), b0, two, false)};
                    G.job_begin();
                    G.term<2>(db, false, pu, p, {0u, 64u});
                    G.job_end([&](uint32_t t) {
                        const int bl = b0 + (row >> 6), tok = 16 * grp;
                        const bool ok = row < 64 || two;
                        float x[16], y[16], act[16];
                        acc16(t + tok, x);
                        acc16(t + 64 + tok, y);
                        if (ok) {
                            ld_split16(sblk(tl.sAk) + ((size_t)bl * tb + tk) * B, row & 63, tok, act);
                            float* akb = ws + tl.bakb + (((size_t)bl * tb + tk) * 64 + tok) * 64 + (row & 63);
                            const float* kw = sh.kw + tk * 64 + tok;
                            const float* km = sh.km + tk * 64 + tok;
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                akb[64 * j] = -(kw[j] * x[j] + km[j] * y[j]);
                                x[j] *= act[j];
                                y[j] *= act[j];
                            }
                        } else {
#pragma unroll
                            for (int j = 0; j < 16; ++j) x[j] = y[j] = 0.0f;
                        }
                        kwb -= reduce16(x, lane);
                        kmb -= reduce16(y, lane);
                    });
                }
            }
            if (G.epi() && (lane & 1) == 0) {
                sh.red[tk][q4][16 * grp + (lane >> 1)][0] = kwb;
                sh.red[tk][q4][16 * grp + (lane >> 1)][1] = kmb;
            }
            // shares of pub = -(K^W T_last a + K^M S_last a) + .. and of dk = -(K^W T_first^T pz + K^M S_first^T pz) + ..
            auto scaled = [&](size_t base) {
                return [&, base](uint32_t t) {
                    const int tok = 16 * grp;
                    float x[16], y[16];
                    acc16(t + tok, x);
                    acc16(t + 64 + tok, y);
                    float* out = partial(base, 0, tk) + (size_t)tok * dp + row;
                    const float* kw = sh.kw + tk * 64 + tok;
                    const float* km = sh.km + tk * 64 + tok;
                    if (row < dp)
#pragma unroll
                        for (int j = 0; j < 16; ++j) out[(size_t)j * dp] = -(kw[j] * x[j] + km[j] * y[j]);
                };
            };
            {
                const Opnd p[2] = {by_d(blk(tl.Tb[LAST]), false), by_d(blk(tl.Sb[LAST]), false)};
                G.job_begin();
                G.term<2>(nsl, false, tok_h(sblk(tl.sAk), tk), p, {0u, 64u});
                G.job_end(scaled(tl.bslot));
            }
            G.job_begin();
#pragma unroll
            for (int i = 0; i < LAST; ++i) {
                const Opnd p[2] = {by_d(blk(tl.Tb[i]), true), by_d(blk(tl.Sb[i]), true)};
                G.term<2>(nsl, false, tok_h(sblk(tl.sPz[i]), tk), p, {0u, 64u});
            }
            G.job_end(scaled(tl.bdk[buf]));
        }
        G.sync_cta();

        // the CTA's share of the adjoints of K^W_t, K^M_t
        for (int e = threadIdx.x; e < tbn * 128; e += kThreads) {
            const int t = e >> 1, w = e & 1;
            float x = 0.0f;
#pragma unroll
            for (int i = 0; i < 4; ++i) x += sh.red[t >> 6][i][t & 63][w];
            sl[tl.skwb + ((size_t)w * kTileShares + rank) * tb * 64 + t] = x;
        }
        // pub += W_last phb
        for (int tk = 0; tk < tbn; ++tk) {
            const Opnd p[1] = {by_d(sblk(tl.sW[LAST]), false)};
            G.job_begin();
            G.term<1>(nsl, false, tok_h(blk(tl.bPhb), tk), p, {0u});
            G.job_end([&](uint32_t t) {
                const int tok = 16 * grp;
                float x[16];
                acc16(t + tok, x);
                float* out = partial(tl.bslot, 1, tk) + (size_t)tok * dp + row;
                if (row < dp)
#pragma unroll
                    for (int j = 0; j < 16; ++j) out[(size_t)j * dp] = x[j];
            });
        }
        G.sync_cluster();

        // ---- rows: pu = J(u) e, e = k + y - v, y = LN(u): adjoints of e and u; dv --------------------------------------------------
        if (G.epi()) {
            const int ci = 4 * lane;
            __nv_bfloat16* dvc = reinterpret_cast<__nv_bfloat16*>(a.dv) + ((size_t)seq * a.Ls + s) * d;
            for (int t = rank * kEpiWarps + warp; t < tbn * 64; t += CL * kEpiWarps) {
                float ub[4] = {0.f, 0.f, 0.f, 0.f};
                if (t < len) {
                    float pub[4] = {0.f, 0.f, 0.f, 0.f}, y[4] = {0.f, 0.f, 0.f, 0.f}, pu[4] = {0.f, 0.f, 0.f, 0.f}, eb[4], ng[4];
                    const float r = sl[tl.sr + t], mey = sl[tl.smey + t], inv = 1.0f / (float)d;
                    if (ci < dp) {
                        const float4 y4 = *reinterpret_cast<const float4*>(sl + tl.sy + (size_t)t * dp + ci);
                        const float4 p4 = *reinterpret_cast<const float4*>(sl + tl.spu + (size_t)t * dp + ci);
                        y[0] = y4.x; y[1] = y4.y; y[2] = y4.z; y[3] = y4.w;
                        pu[0] = p4.x; pu[1] = p4.y; pu[2] = p4.z; pu[3] = p4.w;
                        add_parts(ws + tl.bslot + (size_t)t * dp + ci, 2 * CL, (size_t)tb * 64 * dp, pub);
                    }
                    const float sx = warp_sum(sum4(pub)) * inv, mpy = warp_sum(dot4(pub, y)) * inv, spp = warp_sum(dot4(pub, pu));
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        eb[j] = ci + j < d ? r * (pub[j] - sx - y[j] * mpy) : 0.0f;
                        ng[j] = -eb[j];
                    }
                    const float s2 = warp_sum(sum4(eb)) * inv, s2y = warp_sum(dot4(eb, y)) * inv;
                    // second-order term of the LN Jacobian, and dy -> du for the y inside e
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        ub[j] = ci + j < d ? r * (eb[j] - s2 - y[j] * s2y) - r * inv * spp * y[j] - r * (mpy * pu[j] + mey * eb[j]) : 0.0f;
                    st_tok4(dvc + (size_t)t * d, ci, d, ng);
                    if (ci < dp) *reinterpret_cast<float4*>(ws + tl.bEb[buf] + (size_t)t * dp + ci) = make_float4(eb[0], eb[1], eb[2], eb[3]);
                }
                if (ci < dp) st_split4<true>(blk(tl.bUk) + (size_t)((t >> 6) * db + (lane >> 4)) * B, t & 63, ci & 63, ub);
            }
            if (g + 1 < ga.ng) finish_dk(c + 1, buf ^ 1);
        }
        G.sync_cluster();

        // ---- u = W_last a ; a = act(z): adjoint of z ---------------------------------------------------------------------------
        for (int tk = 0; tk < tbn; ++tk)
            for (int b0 = hb0; b0 < hb1; b0 += 2) {
                const bool two = b0 + 1 < hb1;
                const Opnd uk{blk(tl.bUk) + (size_t)tk * db * B, nullptr, B, true, false};
                const Opnd p[1] = {by_h(sblk(tl.sW[LAST]), b0, two, false)};
                G.job_begin();
                G.term<1>(db, false, uk, p, {0u});
                G.job_end([&](uint32_t t) {
                    const int bl = b0 + (row >> 6), tok = 16 * grp;
                    float x[16], z[16], cv[16], ab[16];
                    const bool ok = row < 64 || two;
                    const size_t e0 = (((size_t)bl * tb + tk) * 64 + tok) * 64 + (row & 63);
                    if (ok)
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            ab[j] = ws[tl.bakb + e0 + 64 * j];
                            z[j] = ws[tl.bz0[0] + e0 + 64 * j];
                            cv[j] = sl[tl.sc1 + e0 + 64 * j];
                        }
                    acc16(t + tok, x);
                    if (!ok) return;
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        x[j] += ab[j];
                        z[j] += x[j] * cv[j];
                    }
                    if (SW)
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            ab[j] = ws[tl.bz0[LAST - 1] + e0 + 64 * j];
                            cv[j] = sl[tl.sc2 + e0 + 64 * j];
                        }
                    st_split16(blk(tl.bZk[0]) + ((size_t)bl * tb + tk) * B, row & 63, tok, z);
                    if (SW) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) ab[j] += x[j] * cv[j];
                        st_split16(blk(tl.bZk[LAST - 1]) + ((size_t)bl * tb + tk) * B, row & 63, tok, ab);
                    }
                });
            }
        G.sync_cta();

        // ---- dk += W_first^T zb: the CTA's share --------------------------------------------------------------------------------
        for (int tk = 0; tk < tbn; ++tk) {
            G.job_begin();
#pragma unroll
            for (int i = 0; i < LAST; ++i) {
                const Opnd p[1] = {by_d(sblk(tl.sW[i]), true)};
                G.term<1>(nsl, false, tok_h(blk(tl.bZk[i]), tk), p, {0u});
            }
            G.job_end([&](uint32_t t) {
                const int tok = 16 * grp;
                float x[16];
                acc16(t + tok, x);
                float* out = partial(tl.bdk[buf], 1, tk) + (size_t)tok * dp + row;
                if (row < dp)
#pragma unroll
                    for (int j = 0; j < 16; ++j) out[(size_t)j * dp] = x[j];
            });
        }

        // ---- adjoints of the chunk-start state: T' = cw T + (adjoint through the chunk), S' = cm T + cb S; carries' adjoints ----------
        {
            const float cw = sc.cw, cm = sc.cm, cb = sc.cb;
            float pw = 0.0f, pm = 0.0f, pb = 0.0f;
            auto transition = [&](int i, size_t e0, size_t es, bool lane_ok, int nj, uint32_t t, unsigned char* tbk, unsigned char* sbk, int brow,
                                  int bcol) {
                float *T = ws + lay.T[i] + e0, *S = ws + lay.S[i] + e0;
                const float *W = ck + (size_t)i * dh + e0, *M = ck + (size_t)(NMAT + i) * dh + e0;
                float tn[16], sn[16];
                acc16(t, tn);
#pragma unroll
                for (int j0 = 0; j0 < 16; j0 += 8) {
                    float tv[8], sv[8], wv[8], mv[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const bool ok = lane_ok && j0 + j < nj;
                        const size_t e = (size_t)(j0 + j) * es;
                        tv[j] = ok ? T[e] : 0.0f; sv[j] = ok ? S[e] : 0.0f;
                        wv[j] = ok ? W[e] : 0.0f; mv[j] = ok ? M[e] : 0.0f;
                    }
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const bool ok = lane_ok && j0 + j < nj;
                        const size_t e = (size_t)(j0 + j) * es;
                        pw += tv[j] * wv[j]; pm += tv[j] * mv[j]; pb += sv[j] * mv[j];
                        tn[j0 + j] = ok ? cw * tv[j] + tn[j0 + j] : 0.0f;
                        sn[j0 + j] = cm * tv[j] + cb * sv[j];
                        if (ok) { T[e] = tn[j0 + j]; S[e] = sn[j0 + j]; }
                    }
                }
                if (tbk) {
                    if (!normed) st_split16(tbk, brow, bcol, tn);
                    st_split16(sbk, brow, bcol, sn);
                }
            };
            for (int b0 = hb0; b0 < hb1; b0 += 2) {
                const bool two = b0 + 1 < hb1;
                auto h_tok = [&](const unsigned char* m) {  // [h x tokens] with contraction over the tokens
                    const unsigned char* p = m + (size_t)b0 * tb * B;
                    return Opnd{p, two ? p + (size_t)tb * B : nullptr, B, true, false};
                };
#pragma unroll
                for (int i = 0; i < LAST; ++i) {
                    const unsigned char *kb = sblk(tl.sK), *qb = sblk(tl.sQ);
                    const Opnd kt{kb, db == 2 ? kb + kHalf : nullptr, (uint32_t)db * kHalf, false, true};
                    const Opnd qt{qb, db == 2 ? qb + kHalf : nullptr, (uint32_t)db * kHalf, false, true};
                    const Opnd pq[1] = {h_tok(sblk(tl.sZq[i]))}, pk[1] = {h_tok(blk(tl.bZk[i]))};
                    G.job_begin();
                    G.term<1>(tbn, true, qt, pq, {0u});
                    G.term<1>(tbn, true, kt, pk, {0u});
                    G.job_end([&](uint32_t t) {
#pragma unroll 1
                        for (int half = 0; half < 2; ++half) {
                            const int col = 32 * grp + 16 * half, j0 = b0 * 64 + col;
                            if (col >= 64 && !two) break;
                            const size_t bo = ((size_t)(b0 + (col >> 6)) * db + (row >> 6)) * B;
                            const bool in = row < dp;
                            transition(i, (size_t)j0 * d + row, d, row < d, h - j0, t + col, in ? blk(tl.Tb[i]) + bo : nullptr,
                                       in ? blk(tl.Sb[i]) + bo : nullptr, row & 63, col & 63);
                        }
                    });
                }
                {
                    auto tok_d = [&](const unsigned char* m) { return Opnd{m, db == 2 ? m + B : nullptr, (uint32_t)db * B, true, true}; };
                    const Opnd u0[1] = {tok_d(sblk(tl.sUq))}, u1[1] = {tok_d(sblk(tl.sPu))}, u2[1] = {tok_d(blk(tl.bUk))};
                    G.job_begin();
                    G.term<1>(tbn, true, h_tok(sblk(tl.sAq)), u0, {0u});
                    G.term<1>(tbn, true, h_tok(blk(tl.bPhb)), u1, {0u});
                    G.term<1>(tbn, true, h_tok(sblk(tl.sAk)), u2, {0u});
                    G.job_end([&](uint32_t t) {
                        const int bl = b0 + (row >> 6), j = b0 * 64 + row;
                        const bool in = row < 64 || two;
#pragma unroll 1
                        for (int half = 0; half < 2; ++half) {
                            const int col = 32 * grp + 16 * half;
                            if (col >= dp) break;
                            const size_t bo = ((size_t)bl * db + (col >> 6)) * B;
                            transition(LAST, (size_t)col * h + j, h, in && j < h, d - col, t + col, in ? blk(tl.Tb[LAST]) + bo : nullptr,
                                       in ? blk(tl.Sb[LAST]) + bo : nullptr, row & 63, col & 63);
                        }
                    });
                }
            }
            if (G.epi()) {
                pw = warp_sum(pw); pm = warp_sum(pm); pb = warp_sum(pb);
                if (lane == 0) { sh.dots[warp][0] = pw; sh.dots[warp][1] = pm; sh.dots[warp][2] = pb; }
            }
        }
        G.sync_cta();
        if (threadIdx.x < 3) {
            float x = 0.0f;
            for (int w = 0; w < kEpiWarps; ++w) x += sh.dots[w][threadIdx.x];
            sl[tl.sdots + rank * 4 + threadIdx.x] = x;
        }
    }
    G.sync_cluster();
    if (G.epi()) {
        finish_dk(ga.c0, ga.c0 & 1);
        if (ga.last && !a.carry_out) {
#pragma unroll
            for (int i = 0; i < NMAT; ++i) {
                float *wf = a.dW_init[i] + (size_t)seq * dh, *mf = a.dM_init[i] + (size_t)seq * dh;
                const float *T = ws + lay.T[i], *S = ws + lay.S[i];
                batched_for<8>(threadIdx.x + (size_t)rank * kEpiThreads, dh, (size_t)kEpiThreads * CL,
                               [&](size_t e) { return make_float2(T[e], S[e]); }, [&](size_t e, const float2& x) { wf[e] = x.x; mf[e] = x.y; });
            }
        }
    }
    G.teardown();
}

// ---- reverse of the suffix scans -------------------------------------------------------------------------------------------------
// One thread walks the chunk (a 3-term linear recurrence, ~10 flop per token) over operands in shared memory; the chunks are
// independent.
__global__ void __launch_bounds__(128) tile_gate_kernel(const GroupArgs ga) {
    __shared__ float in[8][kMaxC], res[3][kMaxC];
    const SimtBwdArgs& a = ga.a;
    const TileLayout& tl = a.lay.tl;
    const int seq = blockIdx.x / ga.ng, g = blockIdx.x % ga.ng, c = ga.c0 + g, s = c * a.C, len = min(a.C, a.L - s), CL = a.cl;
    const float* sl = slot_of(a, seq, ga.s0 + g);
    const ChunkScalars<float>& sc = *reinterpret_cast<const ChunkScalars<float>*>(sl + tl.ssc);
    const size_t t0 = (size_t)seq * a.Ls + s;
    for (int t = threadIdx.x; t < len; t += blockDim.x) {
        in[0][t] = a.beta[t0 + t]; in[1][t] = a.gamma[t0 + t]; in[2][t] = a.eta[t0 + t];
        in[5][t] = sc.S[t + 1]; in[6][t] = sc.bt[t + 1]; in[7][t] = sc.gt[t + 1];
        float w = 0.0f, m = 0.0f;
        for (int r = 0; r < ga.shares; ++r) {
            w += sl[tl.skwb + (size_t)r * tl.tb * 64 + t];
            m += sl[tl.skwb + (size_t)(kTileShares + r) * tl.tb * 64 + t];
        }
        in[3][t] = w; in[4][t] = m;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float gtb = 0.0f, cmb = 0.0f, btb = 0.0f, Sb = 0.0f;
        for (int r = 0; r < CL; ++r) { gtb += sl[tl.sdots + 4 * r]; cmb += sl[tl.sdots + 4 * r + 1]; btb += sl[tl.sdots + 4 * r + 2]; }
        for (int t = 0; t < len; ++t) {
            // index t: state t; token t + 1 lives at array index t
            const float b1 = in[0][t], g1 = in[1][t], e1 = in[2][t], kWb = in[3][t], kMb = in[4][t];
            const float S1 = in[5][t], bt1 = in[6][t], gt1 = in[7][t];
            // S_t = beta_{t+1} S_{t+1} + gt_t ; bt_t = beta_{t+1} bt_{t+1} ; gt_t = gamma_{t+1} gt_{t+1}
            gtb += Sb;
            float bb = Sb * S1 + btb * bt1, Sn = Sb * b1, bn = btb * b1;
            const float gb = gtb * gt1, gn = gtb * g1;
            if (t == 0) { bb += cmb * S1; Sn += cmb * b1; }  // cm = beta_1 S_1
            // K^M_{t+1} = eta bt_{t+1}, K^W_{t+1} = eta S_{t+1}
            res[0][t] = kMb * bt1 + kWb * S1;
            bn += kMb * e1;
            Sn += kWb * e1;
            res[1][t] = bb;
            res[2][t] = gb;
            Sb = Sn; btb = bn; gtb = gn;
        }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < len; t += blockDim.x) {
        a.d_eta[t0 + t] = res[0][t];
        a.d_beta[t0 + t] = res[1][t];
        a.d_gamma[t0 + t] = res[2][t];
    }
}

constexpr size_t kRevSmem = kRecSmem + sizeof(RevShared);

template <int KIND> cudaError_t launch_rev(const GroupArgs& ga, cudaStream_t st) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(ga.a.N * ga.a.cl));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kRevSmem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)ga.a.cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, tile_rev_kernel<KIND>, ga);
}

template <int KIND> int launch(const SimtBwdArgs& a0, cudaStream_t st) {
    static bool attr_done[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return (int)cudaGetLastError();
    if (dev < 0 || dev >= 64 || !attr_done[dev]) {
        cudaError_t e = cudaFuncSetAttribute(tile_rec_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRecSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(tile_rev_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRevSmem);
        if (e != cudaSuccess) return (int)e;
        if (dev >= 0 && dev < 64) attr_done[dev] = true;
    }
    GroupArgs ga{};
    ga.a = a0;
    const TileLayout& tl = a0.lay.tl;
    ga.a.cl = tile_chain_serves(tl) ? tile_chain_ctas(tl) : tl.cl;
    ga.shares = tile_chain_serves(tl) ? 4 * ga.a.cl : tl.cl;
    auto prep = [&](const GroupArgs& g) {  // chunks of up to 64 tokens: tile_rec does it
        const int chunks = a0.N * g.ng;
        if (tl.tb > 1) tile_prep_kernel<KIND == 0 ? 2 : 3><<<dim3(chunks, chunks >= 592 ? 1 : (592 + chunks - 1) / chunks), 256, 0, st>>>(g);
    };
    bool have = false;  // this group's tile_rec ran with the chain of the group before
    for (int end = a0.nchunks, n = 0; end > 0; end -= tl.G, ++n) {
        ga.c0 = end > tl.G ? end - tl.G : 0;
        ga.ng = end - ga.c0;
        ga.s0 = tl.sets == 2 && (n & 1) ? tl.G : 0;
        ga.first = end == a0.nchunks;
        ga.last = ga.c0 == 0;
        const int chunks = a0.N * ga.ng, items = chunks * tl.tb;
        if (!have) {
            prep(ga);
            tile_rec_kernel<KIND><<<items < 148 ? items : 148, kThreads, kRecSmem, st>>>(ga);
        }
        NextGroup next{};
        int rec_ctas = 0;
        if (tl.sets == 2 && !ga.last) {
            GroupArgs gn = ga;
            gn.c0 = ga.c0 > tl.G ? ga.c0 - tl.G : 0;
            gn.ng = ga.c0 - gn.c0;
            gn.s0 = ga.s0 ? 0 : tl.G;
            prep(gn);
            next = NextGroup{gn.c0, gn.ng, gn.s0};
            const int want = (a0.N * gn.ng * tl.tb + ga.a.cl - 1) / ga.a.cl * ga.a.cl;
            rec_ctas = want < tl.spare ? want : tl.spare;
        }
        have = rec_ctas > 0;
        cudaError_t e = tile_chain_serves(tl) ? (cudaError_t)tile_chain_launch(ga, next, rec_ctas, KIND, st) : launch_rev<KIND>(ga, st);
        if (e != cudaSuccess) return (int)e;
        tile_gate_kernel<<<chunks, 128, 0, st>>>(ga);
        e = cudaGetLastError();
        if (e != cudaSuccess) return (int)e;
    }
    return 0;
}

}  // namespace

int tile_bwd_launch(const SimtBwdArgs& a, int kind, void* stream) {
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    return kind == 0 ? launch<0>(a, st) : launch<1>(a, st);
}

}  // namespace e2ttt
