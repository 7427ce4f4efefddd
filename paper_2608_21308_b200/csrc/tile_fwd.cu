// Forward on the block-tiled engine (tile.cuh): Algorithm 1 chunk after chunk, bf16 I/O, d <= 128, any h and C, both networks; a few sequences of wide
// networks (tile_flow_serves, tile_flow.h: the others run on work items, tile_flow.cu).
//
// A cluster of up to 8 CTAs works on one sequence; CTA r owns a slice of the hidden units - its rows of the first matrices, its
// columns of the last - and computes everything that lives on hidden units for its slice alone.  What is summed over hidden
// units (u = W_last a, [tokens x d]) is left in the workspace as one partial sum per CTA; after a cluster barrier every CTA adds
// the parts of its share of the rows in CTA order and runs the layer norm and its adjoint on them.
// State: fp32, row-major, in the workspace (or directly in the slots of the saved states), updated by the aggregation's epilogue, which
// also writes the operand blocks of the next chunk's weights.
#include "tile.cuh"
#include "tile_flow.h"

namespace e2ttt {
using namespace tile;

namespace {

template <int KIND> __global__ void __launch_bounds__(kThreads, 1) tile_fwd_kernel(const SimtFwdArgs a) {
    constexpr int NMAT = (KIND == 0) ? 2 : 3, LAST = NMAT - 1;
    constexpr bool SW = KIND == 1;
    extern __shared__ unsigned char tile_smem[];
    unsigned char* ring = tile_smem + ((1024u - (smem_u32(tile_smem) & 1023u)) & 1023u);
    Sync* sy = reinterpret_cast<Sync*>(ring + kUnits * kUnitBytes);
    ChunkScalars<float>& sc = *reinterpret_cast<ChunkScalars<float>*>(sy + 1);

    const int CL = a.cl, seq = blockIdx.x / CL, rank = blockIdx.x % CL;
    Engine G;
    G.setup(ring, sy, a.status, rank, CL);
    const int warp = G.warp, lane = G.lane;
    const int q4 = warp & 3, grp = warp >> 2;  // lane quadrant, column quarter
    const int row = 32 * q4 + lane;
    const int d = a.d, h = a.h, C = a.C, L = a.L;
    const size_t dh = (size_t)d * h;
    const SimtLayout& lay = a.lay;
    const TileLayout& tl = lay.tl;
    const int db = tl.db, hb = tl.hb, tb = tl.tb, dp = db * 64;
    const int sb = (hb + CL - 1) / CL, hb0 = min(hb, rank * sb), hb1 = min(hb, hb0 + sb), nsl = hb1 - hb0;
    float* ws = reinterpret_cast<float*>(a.ws) + (size_t)seq * lay.per_seq;
    auto blk = [&](size_t off) { return reinterpret_cast<unsigned char*>(ws + off); };
    const __nv_bfloat16* q = reinterpret_cast<const __nv_bfloat16*>(a.q) + (size_t)seq * a.Ls * d;
    const __nv_bfloat16* k = reinterpret_cast<const __nv_bfloat16*>(a.k) + (size_t)seq * a.Ls * d;
    const __nv_bfloat16* v = reinterpret_cast<const __nv_bfloat16*>(a.v) + (size_t)seq * a.Ls * d;
    __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(a.o) + (size_t)seq * a.Ls * d;
    const float* eta = a.eta + (size_t)seq * a.Ls;
    const float* beta = a.beta + (size_t)seq * a.Ls;
    const float* gamma = a.gamma + (size_t)seq * a.Ls;
    const bool normed = a.row_norm[0] != nullptr;
    constexpr uint32_t B = 2 * kHalf;  // bytes of a block

    // ---- chunk 0: operand blocks of the initial weights and of the tokens; the initial state into the saved slots ------------
    const float* ck0 = a.init_slot >= 0 ? ws + lay.cck + (size_t)a.init_slot * 2 * NMAT * dh : nullptr;
    const float *w_in[NMAT], *m_in[NMAT];
#pragma unroll
    for (int i = 0; i < NMAT; ++i) {
        w_in[i] = ck0 ? ck0 + (size_t)i * dh : a.W_init[i] + (size_t)seq * dh;
        m_in[i] = ck0 ? ck0 + (size_t)(NMAT + i) * dh : (a.M_init[i] ? a.M_init[i] + (size_t)seq * dh : nullptr);
    }
    if (G.epi()) {
#pragma unroll
        for (int i = 0; i < NMAT; ++i) {
            if (i < LAST) matrix_to_blocks(w_in[i], d, h, 0, db, hb0, hb1, blk(tl.Wb[i]), 1, db, warp, kEpiWarps, lane);
            else matrix_to_blocks(w_in[i], h, d, hb0, hb1, 0, db, blk(tl.Wb[i]), db, 1, warp, kEpiWarps, lane);
        }
        tokens_to_blocks(k, min(C, L), d, db, tb, blk(tl.fK[0]), rank * kEpiWarps + warp, CL * kEpiWarps, lane);
        tokens_to_blocks(q, min(C, L), d, db, tb, blk(tl.fQ[0]), rank * kEpiWarps + warp, CL * kEpiWarps, lane);
        if (a.save_states) {
            float* ck = ws + (a.save_states == 1 ? lay.ckpt : lay.cck);
            if (ck != ck0) {
#pragma unroll
                for (int i = 0; i < NMAT; ++i)
                    batched_for<8>(threadIdx.x + (size_t)rank * kEpiThreads, dh, (size_t)kEpiThreads * CL,
                                   [&](size_t e) { return make_float2(w_in[i][e], m_in[i] ? m_in[i][e] : 0.0f); },
                                   [&](size_t e, const float2& x) { ck[i * dh + e] = x.x; ck[(NMAT + i) * dh + e] = x.y; });
            }
        }
    }
    G.sync_cluster();

    for (int c = 0; c < a.nchunks; ++c) {
        const int s = c * C, len = min(C, L - s), tbn = (len + 63) / 64;
        const __nv_bfloat16* kc = k + (size_t)s * d;
        const __nv_bfloat16* qc = q + (size_t)s * d;
        const __nv_bfloat16* vc = v + (size_t)s * d;
        const unsigned char* Kb = blk(tl.fK[c & 1]);
        const unsigned char* Qb = blk(tl.fQ[c & 1]);
        if (warp == 0) chunk_scalars_warp<float>(eta + s, beta + s, gamma + s, len, &sc);  // Algorithm 1 line 2

        // ---- z = W_first x on keys (columns 0-63) and queries (64-127); a = act(z) ------------------------------------------
        for (int tk = 0; tk < tbn; ++tk)
            for (int b0 = hb0; b0 < hb1; b0 += 2) {
                const bool two = b0 + 1 < hb1;
                auto wop = [&](int i) {
                    const unsigned char* p = blk(tl.Wb[i]) + (size_t)b0 * db * B;
                    return Opnd{p, two ? p + (size_t)db * B : nullptr, B, true, true};
                };
                const Opnd x{Kb + (size_t)tk * db * kHalf, Qb + (size_t)tk * db * kHalf, kHalf, false, false};
                G.job_begin();
                if constexpr (SW) {
                    const Opnd w[2] = {wop(0), wop(1)};
                    G.term<2>(db, false, x, w, {0u, 128u});
                } else {
                    const Opnd w[1] = {wop(0)};
                    G.term<1>(db, false, x, w, {0u});
                }
                G.job_end([&](uint32_t t) {
                    const int bl = b0 + (row >> 6);
                    const bool key = grp < 2;
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        const int col = 32 * grp + 16 * half, tok = col & 63;
                        float z1[16], z2[16], act[16];
                        acc16(t + col, z1);
                        if (SW) acc16(t + 128 + col, z2);
                        if (row >= 64 && !two) continue;
                        const size_t e0 = (((size_t)bl * tb + tk) * 64 + tok) * 64 + (row & 63);
                        float* c1 = ws + tl.fc1 + e0;
                        float* c2 = ws + tl.fc2 + e0;
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            if (!SW) {
                                float cdf, pdf;
                                normal_dist(z1[j], cdf, pdf);
                                act[j] = z1[j] * cdf;
                                if (key) c1[64 * j] = cdf + z1[j] * pdf;
                            } else {
                                const float sg = sigmoid_hw(z1[j]), sl = z1[j] * sg;
                                act[j] = sl * z2[j];
                                if (key) {
                                    c1[64 * j] = z2[j] * (sg * (1.0f + z1[j] * (1.0f - sg)));
                                    c2[64 * j] = sl;
                                }
                            }
                        }
                        st_split16(blk(key ? tl.fA : tl.fAq) + ((size_t)bl * tb + tk) * B, row & 63, tok, act);
                    }
                });
            }
        G.sync_cta();

        // ---- u = W_last a over the CTA's hidden units: partial sums ----------------------------------------------------------
        for (int tk = 0; tk < tbn; ++tk) {
            const unsigned char* pw = blk(tl.Wb[LAST]) + (size_t)hb0 * db * B;
            const Opnd act{blk(tl.fA) + ((size_t)hb0 * tb + tk) * B, blk(tl.fAq) + ((size_t)hb0 * tb + tk) * B, (uint32_t)tb * B, true, true};
            const Opnd w[1] = {{pw, db == 2 ? pw + B : nullptr, (uint32_t)db * B, true, true}};
            G.job_begin();
            G.term<1>(nsl, false, act, w, {0u});
            G.job_end([&](uint32_t t) {
                float* slot = ws + tl.fslot + ((size_t)(rank * tb + tk) * 128 + 32 * grp) * dp + row;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    float u[16];
                    acc16(t + 32 * grp + 16 * half, u);
                    if (row < dp)
#pragma unroll
                        for (int j = 0; j < 16; ++j) slot[(size_t)(16 * half + j) * dp] = u[j];
                }
            });
        }
        G.sync_cluster();

        // ---- rows: layer norm; outputs of the queries; pu = dL/du of the keys (Algorithm 1 line 3) ----------------------------
        if (G.epi()) {
            const int ci = 4 * lane, step = CL * kEpiWarps, nrows = tbn * 128;
            constexpr int R = 2;  // rows of a warp in flight: a row is a chain of loads and five reductions
            for (int r0 = rank * kEpiWarps + warp; r0 < nrows; r0 += R * step) {
                float u[R][4], x[R][4], vv[R][4], mu[R], rs[R];
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const int rr = min(r0 + i * step, nrows - 1), t = min((rr >> 7) * 64 + (rr & 63), len - 1);
                    ld_tok4(((rr & 127) < 64 ? kc : qc) + (size_t)t * d, ci, d, x[i]);
                    ld_tok4(vc + (size_t)t * d, ci, d, vv[i]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) u[i][j] = 0.0f;
                }
                for (int r = 0; r < CL; ++r) {  // the CTAs' partial sums, in CTA order
                    float4 p[R];
#pragma unroll
                    for (int i = 0; i < R; ++i)
                        p[i] = *reinterpret_cast<const float4*>(ws + tl.fslot + ((size_t)r * tb * 128 + min(r0 + i * step, nrows - 1)) * dp + min(ci, dp - 4));
#pragma unroll
                    for (int i = 0; i < R; ++i) { u[i][0] += p[i].x; u[i][1] += p[i].y; u[i][2] += p[i].z; u[i][3] += p[i].w; }
                }
#pragma unroll
                for (int i = 0; i < R; ++i) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) u[i][j] = ci + j < d ? u[i][j] : 0.0f;
                    mu[i] = sum4(u[i]);
                }
                warp_sums(mu);
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const float m = mu[i] / (float)d;
#pragma unroll
                    for (int j = 0; j < 4; ++j) u[i][j] = ci + j < d ? u[i][j] - m : 0.0f;
                    rs[i] = dot4(u[i], u[i]);
                }
                warp_sums(rs);
                float se[R], sey[R];
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    rs[i] = r_rsqrt(rs[i] / (float)d + a.eps);
                    float e[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        u[i][j] *= rs[i];
                        e[j] = x[i][j] + u[i][j] - vv[i][j];
                    }
                    se[i] = sum4(e);
                    sey[i] = dot4(e, u[i]);
                }
                warp_sums(se);
                warp_sums(sey);
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const int rr = r0 + i * step, tk = rr >> 7, t = tk * 64 + (rr & 63);
                    if (rr >= nrows) continue;
                    const bool live = t < len;
                    if ((rr & 127) >= 64) {
                        if (live && a.o) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) u[i][j] += x[i][j];
                            st_tok4(o + (size_t)(s + t) * d, ci, d, u[i]);
                        }
                        continue;
                    }
                    const float kw = live ? sc.kW[t] : 0.0f, km = live ? sc.kM[t] : 0.0f;
                    float pu[4], uw[4], um[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float e = x[i][j] + u[i][j] - vv[i][j];
                        pu[j] = live && ci + j < d ? rs[i] * (e - se[i] / (float)d - u[i][j] * (sey[i] / (float)d)) : 0.0f;
                        uw[j] = kw * pu[j];
                        um[j] = km * pu[j];
                    }
                    if (ci < dp) {
                        const size_t off = (size_t)(tk * db + (lane >> 4)) * B;
                        st_split4<true>(blk(tl.fPu) + off, t & 63, ci & 63, pu);
                        st_split4<true>(blk(tl.fPuW) + off, t & 63, ci & 63, uw);
                        st_split4<true>(blk(tl.fPuM) + off, t & 63, ci & 63, um);
                    }
                }
            }
            if (c + 1 < a.nchunks) {  // the next chunk's tokens
                const int n = min(C, L - s - C);
                tokens_to_blocks(kc + (size_t)C * d, n, d, db, tb, blk(tl.fK[(c + 1) & 1]), rank * kEpiWarps + warp, CL * kEpiWarps, lane);
                tokens_to_blocks(qc + (size_t)C * d, n, d, db, tb, blk(tl.fQ[(c + 1) & 1]), rank * kEpiWarps + warp, CL * kEpiWarps, lane);
            }
        }
        G.sync_cluster();

        // ---- back through the last matrix and the activation: K^W pz, K^M pz -----------------------------------------------
        for (int tk = 0; tk < tbn; ++tk)
            for (int b0 = hb0; b0 < hb1; b0 += 2) {
                const bool two = b0 + 1 < hb1;
                const unsigned char* pw = blk(tl.Wb[LAST]) + (size_t)b0 * db * B;
                const Opnd pu{blk(tl.fPu) + (size_t)tk * db * B, nullptr, B, true, false};
                const Opnd w[1] = {{pw, two ? pw + (size_t)db * B : nullptr, B, true, false}};
                G.job_begin();
                G.term<1>(db, false, pu, w, {0u});
                G.job_end([&](uint32_t t) {
                    const int bl = b0 + (row >> 6), tok = 16 * grp;
                    float ph[16], pw16[16], pm16[16];
                    acc16(t + tok, ph);
                    if (row >= 64 && !two) return;
                    const size_t e0 = (((size_t)bl * tb + tk) * 64 + tok) * 64 + (row & 63);
#pragma unroll
                    for (int i = 0; i < LAST; ++i) {
                        const float* cf = ws + (i == 0 ? tl.fc1 : tl.fc2) + e0;
                        float cv[16];
#pragma unroll
                        for (int j = 0; j < 16; ++j) cv[j] = cf[64 * j];
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const int tt = tk * 64 + tok + j;
                            const float p = ph[j] * cv[j];
                            pw16[j] = tt < len ? sc.kW[tt] * p : 0.0f;
                            pm16[j] = tt < len ? sc.kM[tt] * p : 0.0f;
                        }
                        st_split16(blk(tl.fPzW[i]) + ((size_t)bl * tb + tk) * B, row & 63, tok, pw16);
                        st_split16(blk(tl.fPzM[i]) + ((size_t)bl * tb + tk) * B, row & 63, tok, pm16);
                    }
                });
            }
        G.sync_cta();

        // ---- Algorithm 1 lines 4-7: both weighted aggregations of every matrix, fused with the state transition --------------
        const float cw = sc.cw, cm = sc.cm, cb = sc.cb;
        const bool last_chunk = c + 1 == a.nchunks;
        float *w_out[NMAT], *m_out[NMAT], *w_copy[NMAT], *m_copy[NMAT];
#pragma unroll
        for (int i = 0; i < NMAT; ++i) {
            w_out[i] = ws + lay.W[i]; m_out[i] = ws + lay.M[i];
            w_copy[i] = m_copy[i] = nullptr;
            float* fw = a.W_final[i] ? a.W_final[i] + (size_t)seq * dh : nullptr;
            float* fm = a.W_final[i] ? a.M_final[i] + (size_t)seq * dh : nullptr;
            if (a.save_states == 1) {
                float* ck = ws + lay.ckpt + (size_t)(c + 1) * 2 * NMAT * dh;
                w_out[i] = ck + (size_t)i * dh; m_out[i] = ck + (size_t)(NMAT + i) * dh;
                if (last_chunk && fw) { w_copy[i] = fw; m_copy[i] = fm; }
            } else if (last_chunk && fw && !normed) {
                w_out[i] = fw; m_out[i] = fm;
            } else if (a.save_states == 2 && (c + 1) % lay.seg == 0) {
                float* ck = ws + lay.cck + (size_t)((c + 1) / lay.seg) * 2 * NMAT * dh;
                w_copy[i] = ck + (size_t)i * dh; m_copy[i] = ck + (size_t)(NMAT + i) * dh;
            }
        }
        // 16 results of one lane: elements base + ln + j * es, j < nj, of lane index ln < nl; weights' aggregate in columns col..,
        // momentum's 128 further.  Indices are clamped and values masked: with a branch at every load they were one round trip each
        auto transition = [&](int i, size_t base, int ln, int nl, int es, int nj, uint32_t t, int col, unsigned char* wb, int brow) {
            float acc[16], w[16], m[16];
            const bool lane_ok = ln < nl;
            if (nj > 0) {
                const size_t b = base + min(ln, nl - 1);
#pragma unroll
                for (int j = 0; j < 16; ++j) w[j] = w_in[i][b + (size_t)(min(j, nj - 1) * es)];
                if (m_in[i])
#pragma unroll
                    for (int j = 0; j < 16; ++j) m[j] = m_in[i][b + (size_t)(min(j, nj - 1) * es)];
                else
#pragma unroll
                    for (int j = 0; j < 16; ++j) m[j] = 0.0f;
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) w[j] = m[j] = 0.0f;
            }
            acc16(t + 128 + col, acc);  // G_t = -grad: the aggregations enter with a minus sign
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const float mj = m[j];
                m[j] = cb * mj - acc[j];
                w[j] = cw * w[j] + cm * mj;
            }
            acc16(t + col, acc);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const bool ok = lane_ok && j < nj;
                w[j] = ok ? w[j] - acc[j] : 0.0f;
                const size_t e = base + ln + (size_t)(j * es);
                if (ok) {
                    w_out[i][e] = w[j]; m_out[i][e] = m[j];
                    if (w_copy[i]) { w_copy[i][e] = w[j]; m_copy[i][e] = m[j]; }
                }
            }
            if (wb && !normed) st_split16(wb, brow, col & 63, w);
        };
        for (int b0 = hb0; b0 < hb1; b0 += 2) {
            const bool two = b0 + 1 < hb1;
#pragma unroll
            for (int i = 0; i < LAST; ++i) {
                const Opnd kt{Kb, db == 2 ? Kb + kHalf : nullptr, (uint32_t)db * kHalf, false, true};
                auto zop = [&](size_t off) {
                    const unsigned char* p = blk(off) + (size_t)b0 * tb * B;
                    return Opnd{p, two ? p + (size_t)tb * B : nullptr, B, true, false};
                };
                const Opnd pz[2] = {zop(tl.fPzW[i]), zop(tl.fPzM[i])};
                G.job_begin();
                G.term<2>(tbn, true, kt, pz, {0u, 128u});
                G.job_end([&](uint32_t t) {
#pragma unroll 1
                    for (int half = 0; half < 2; ++half) {
                        const int col = 32 * grp + 16 * half, j0 = b0 * 64 + col, bl = b0 + (col >> 6);
                        if (col >= 64 && !two) break;
                        transition(i, (size_t)j0 * d, row, d, d, h - j0, t, col,
                                   row < dp ? blk(tl.Wb[i]) + ((size_t)bl * db + (row >> 6)) * B : nullptr, row & 63);
                    }
                });
            }
            {
                const unsigned char* pa = blk(tl.fA) + (size_t)b0 * tb * B;
                const Opnd act{pa, two ? pa + (size_t)tb * B : nullptr, B, true, false};
                const unsigned char *p0 = blk(tl.fPuW), *p1 = blk(tl.fPuM);
                const Opnd pu[2] = {{p0, db == 2 ? p0 + B : nullptr, (uint32_t)db * B, true, true},
                                    {p1, db == 2 ? p1 + B : nullptr, (uint32_t)db * B, true, true}};
                G.job_begin();
                G.term<2>(tbn, true, act, pu, {0u, 128u});
                G.job_end([&](uint32_t t) {
                    const int bl = b0 + (row >> 6);
#pragma unroll 1
                    for (int half = 0; half < 2; ++half) {
                        const int col = 32 * grp + 16 * half;
                        if (col >= dp) break;
                        transition(LAST, (size_t)col * h + b0 * 64, row, min(two ? 128 : 64, h - b0 * 64), h, d - col, t, col,
                                   row < 64 || two ? blk(tl.Wb[LAST]) + ((size_t)bl * db + (col >> 6)) * B : nullptr, row & 63);
                    }
                });
            }
        }
#pragma unroll
        for (int i = 0; i < NMAT; ++i) { w_in[i] = w_out[i]; m_in[i] = m_out[i]; }

        if (normed) {
            // every row w of every W_i becomes n w / (||w|| + eps_n), one warp per row; then the operand blocks of the result
            G.sync_cluster();
            if (G.epi()) {
                const int maxdim = d > h ? d : h;
                int first = rank * kEpiWarps + warp;
#pragma unroll
                for (int i = 0; i < NMAT; ++i) {
                    const int rows = (i == LAST) ? d : h, cols = (i == LAST) ? h : d;
                    const float* target = a.row_norm[i] + (size_t)seq * rows;
                    for (int r = first; r < rows; r += CL * kEpiWarps) {
                        float* w = w_out[i] + (size_t)r * cols;
                        float ss = 0.0f;
                        for (int j = lane; j < cols; j += 32) ss += w[j] * w[j];
                        const float nrm = sqrtf(warp_sum(ss)), f = target[r] / (nrm + a.norm_eps);
                        for (int j = lane; j < cols; j += 32) {
                            w[j] *= f;
                            if (w_copy[i]) w_copy[i][(size_t)r * cols + j] = w[j];
                        }
                        if (a.save_states && lane == 0) ws[lay.rown + ((size_t)c * 3 + i) * maxdim + r] = nrm;
                    }
                }
            }
            G.sync_cluster();
            if (G.epi() && !last_chunk) {
#pragma unroll
                for (int i = 0; i < NMAT; ++i) {
                    if (i < LAST) matrix_to_blocks(w_out[i], d, h, 0, db, hb0, hb1, blk(tl.Wb[i]), 1, db, warp, kEpiWarps, lane);
                    else matrix_to_blocks(w_out[i], h, d, hb0, hb1, 0, db, blk(tl.Wb[i]), db, 1, warp, kEpiWarps, lane);
                }
            }
            if (G.epi() && last_chunk && a.save_states != 1) {
#pragma unroll
                for (int i = 0; i < NMAT; ++i) {
                    if (!a.W_final[i]) continue;
                    batched_for<8>(threadIdx.x + (size_t)rank * kEpiThreads, dh, (size_t)kEpiThreads * CL,
                                   [&](size_t e) { return make_float2(w_out[i][e], m_out[i][e]); },
                                   [&](size_t e, const float2& x) { a.W_final[i][seq * dh + e] = x.x; a.M_final[i][seq * dh + e] = x.y; });
                }
            }
        }
        G.sync_cta();
    }
    G.sync_cluster();
    G.teardown();
}

constexpr size_t kFwdSmem = 1024 + (size_t)kUnits * kUnitBytes + sizeof(Sync) + sizeof(ChunkScalars<float>);

template <int KIND> int launch(const SimtFwdArgs& a, cudaStream_t st) {
    static bool attr_done[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return (int)cudaGetLastError();
    if (dev < 0 || dev >= 64 || !attr_done[dev]) {
        cudaError_t e = cudaFuncSetAttribute(tile_fwd_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFwdSmem);
        if (e != cudaSuccess) return (int)e;
        if (dev >= 0 && dev < 64) attr_done[dev] = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(a.N * a.lay.tl.cl));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kFwdSmem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)a.lay.tl.cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    SimtFwdArgs b = a;
    b.cl = a.lay.tl.cl;
    cudaError_t e = cudaLaunchKernelEx(&cfg, tile_fwd_kernel<KIND>, b);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaGetLastError();
}

}  // namespace

int tile_fwd_launch(const SimtFwdArgs& a, int kind, void* stream) {
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (tile_flow_serves(a.lay.tl, a.N, a.C, a.Ls, kind == 0 ? 2 : 3, a.row_norm[0] != nullptr)) return tile_flow_launch(a, kind, stream);
    return kind == 0 ? launch<0>(a, st) : launch<1>(a, st);
}

}  // namespace e2ttt
