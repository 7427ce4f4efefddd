// The part of the block-tiled reverse pass that does not depend on the adjoints of the state (tile_bwd.cu), shared by the kernel of its
// own and the chain kernel, whose launch takes the next group's part along on SMs that the chain does not fill (tile_chain.cu).
#pragma once
#include "tile_chain.h"

namespace e2ttt {
namespace tile {

constexpr size_t kRecSmem = 1024 + (size_t)kUnits * kUnitBytes + sizeof(Sync);

// ---- operand blocks of the chunk-start weights and of the tokens; scalar kernels: warp w of nw ------------------------------
template <int NMAT> __device__ __forceinline__ void prepare_chunk(const SimtBwdArgs& a, int seq, int c, float* sl, int w, int nw, int lane) {
    const SimtLayout& lay = a.lay;
    const TileLayout& tl = lay.tl;
    const int d = a.d, h = a.h, s = c * a.C, len = min(a.C, a.L - s);
    const size_t dh = (size_t)d * h;
    const float* ck = reinterpret_cast<const float*>(a.ws) + (size_t)seq * lay.per_seq + lay.ckpt + (size_t)c * 2 * NMAT * dh;
#pragma unroll
    for (int i = 0; i < NMAT; ++i) {
        if (i < NMAT - 1) matrix_to_blocks(ck + i * dh, d, h, 0, tl.db, 0, tl.hb, bytes_of(sl + tl.sW[i]), 1, tl.db, w, nw, lane);
        else matrix_to_blocks(ck + i * dh, h, d, 0, tl.hb, 0, tl.db, bytes_of(sl + tl.sW[i]), tl.db, 1, w, nw, lane);
    }
    const size_t tok = ((size_t)seq * a.Ls + s) * d;
    tokens_to_blocks(reinterpret_cast<const __nv_bfloat16*>(a.k) + tok, len, d, tl.db, tl.tb, bytes_of(sl + tl.sK), w, nw, lane);
    tokens_to_blocks(reinterpret_cast<const __nv_bfloat16*>(a.q) + tok, len, d, tl.db, tl.tb, bytes_of(sl + tl.sQ), w, nw, lane);
    if (w == nw - 1) {
        const size_t t = (size_t)seq * a.Ls + s;
        chunk_scalars_warp<float>(a.eta + t, a.beta + t, a.gamma + t, len, reinterpret_cast<ChunkScalars<float>*>(sl + tl.ssc));
    }
}

// ---- what does not depend on T and S -------------------------------------------------------------------------------------------
// Items (sequence, chunk, 64 tokens) first, first + step, .. of the chunks [c0, c0 + ng), slots from s0
template <int KIND> __device__ __forceinline__ void rec_items(const SimtBwdArgs& a, const NextGroup& ga, unsigned char* tile_smem, int first, int step) {
    constexpr int NMAT = (KIND == 0) ? 2 : 3, LAST = NMAT - 1;
    constexpr bool SW = KIND == 1;
    unsigned char* ring = tile_smem + ((1024u - (smem_u32(tile_smem) & 1023u)) & 1023u);
    Sync* sy = reinterpret_cast<Sync*>(ring + kUnits * kUnitBytes);
    Engine G;
    G.setup(ring, sy, a.status, 0, 1);
    const int warp = G.warp, lane = G.lane, q4 = warp & 3, grp = warp >> 2, row = 32 * q4 + lane;
    const TileLayout& tl = a.lay.tl;
    const int d = a.d, db = tl.db, hb = tl.hb, tb = tl.tb, dp = db * 64;

    const int items = a.N * ga.ng * tb;
    for (int item = first; item < items; item += step) {
        const int tk = item % tb, g = (item / tb) % ga.ng, seq = item / (tb * ga.ng), c = ga.c0 + g;
        const int s = c * a.C, len = min(a.C, a.L - s);
        if (tk * 64 >= len) continue;
        float* sl = slot_of(a, seq, ga.s0 + g);
        if (tb == 1) {  // one item per chunk: its operand blocks are made here, and read while L2 has them
            if (G.epi()) prepare_chunk<NMAT>(a, seq, c, sl, warp, kEpiWarps, lane);
            G.sync_cta();
        }
        auto blk = [&](size_t off) { return bytes_of(sl + off); };
        const size_t tok0 = ((size_t)seq * a.Ls + s) * d;
        const __nv_bfloat16* kc = reinterpret_cast<const __nv_bfloat16*>(a.k) + tok0;
        const __nv_bfloat16* vc = reinterpret_cast<const __nv_bfloat16*>(a.v) + tok0;
        const __nv_bfloat16* doc = reinterpret_cast<const __nv_bfloat16*>(a.d_o) + tok0;
        __nv_bfloat16* dqc = reinterpret_cast<__nv_bfloat16*>(a.dq) + tok0;

        // z = W_first x on the keys (columns 0-63) and queries (64-127); a = act(z) and the activation's derivatives
        for (int b0 = 0; b0 < hb; b0 += 2) {
            const bool two = b0 + 1 < hb;
            auto wop = [&](int i) {
                const unsigned char* p = blk(tl.sW[i]) + (size_t)b0 * db * B;
                return Opnd{p, two ? p + (size_t)db * B : nullptr, B, true, true};
            };
            const Opnd x{blk(tl.sK) + (size_t)tk * db * kHalf, blk(tl.sQ) + (size_t)tk * db * kHalf, kHalf, false, false};
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
#pragma unroll 1
                for (int half = 0; half < 2; ++half) {
                    const int col = 32 * grp + 16 * half, tok = col & 63;
                    float z1[16], z2[16], act[16];
                    acc16(t + col, z1);
                    if (SW) acc16(t + 128 + col, z2);
                    if (row >= 64 && !two) continue;
                    const size_t e0 = (((size_t)bl * tb + tk) * 64 + tok) * 64 + (row & 63);
                    float* c1 = sl + (key ? tl.sc1 : tl.sc1q) + e0;
                    float* c2 = sl + (key ? tl.sc2 : tl.sc2q) + e0;
                    float* c4 = sl + tl.sc4 + e0;
                    float* g1 = sl + tl.sg1 + e0;
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float z = z1[j];
                        if (!SW) {
                            const float cdf = norm_cdf(z), pdf = norm_pdf(z);
                            act[j] = z * cdf;
                            c1[64 * j] = cdf + z * pdf;
                            if (key) c4[64 * j] = pdf * (2.0f - z * z);
                        } else {
                            const float sg = sigmoid_f(z), slu = z * sg, d1 = sg * (1.0f + z * (1.0f - sg));
                            act[j] = slu * z2[j];
                            c1[64 * j] = z2[j] * d1;
                            c2[64 * j] = slu;
                            if (key) {
                                g1[64 * j] = d1;
                                c4[64 * j] = z2[j] * (sg * (1.0f - sg) * (2.0f + z * (1.0f - 2.0f * sg)));
                            }
                        }
                    }
                    st_split16(blk(key ? tl.sAk : tl.sAq) + ((size_t)bl * tb + tk) * B, row & 63, tok, act);
                }
            });
        }
        G.sync_cta();

        // u = W_last a.  One CTA contracts all hidden units: with the small terms apart the chain of truncating MMAs is a third as long
        // (h = 1100, C = 16: error of the gate adjoints against 64 bits 1.17-1.33 -> 1.04-1.17 times that of fp32 sums over eight CTAs;
        // d = 64, h = 1024: of dW 1.13 -> 0.95 times)
        float* U = sl + tl.sU + (size_t)tk * 128 * dp;
        {
            const unsigned char* pw = blk(tl.sW[LAST]);
            const Opnd act{blk(tl.sAk) + (size_t)tk * B, blk(tl.sAq) + (size_t)tk * B, (uint32_t)tb * B, true, true};
            const Opnd w[1] = {{pw, db == 2 ? pw + B : nullptr, (uint32_t)db * B, true, true}};
            G.job_begin();
            G.term<1, true>(hb, false, act, w, {0u});
            G.job_end([&](uint32_t t) {
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const int col = 32 * grp + 16 * half;
                    float u[16], ul[16];
                    acc16(t + col, u);
                    acc16(t + 128 + col, ul);
#pragma unroll
                    for (int j = 0; j < 16; ++j) u[j] += ul[j];
                    if (row < dp)
#pragma unroll
                        for (int j = 0; j < 16; ++j) U[(size_t)(col + j) * dp + row] = u[j];
                }
            });
        }
        G.sync_cta();

        // rows: layer norm; keys: e = k + y - v, pu = J e; queries: the adjoint of the output's layer norm
        if (G.epi()) {
            const int ci = 4 * lane;
            for (int rr = warp; rr < 128; rr += kEpiWarps) {
                const int t = tk * 64 + (rr & 63);
                const bool key = rr < 64, live = t < len;
                float u[4] = {0.f, 0.f, 0.f, 0.f}, out[4] = {0.f, 0.f, 0.f, 0.f};
                if (live) {
                    float x[4], vv[4];
                    ld_tok4((key ? kc : doc) + (size_t)t * d, ci, d, x);
                    if (key) ld_tok4(vc + (size_t)t * d, ci, d, vv);
                    if (ci < dp) {
                        const float4 p = *reinterpret_cast<const float4*>(U + (size_t)rr * dp + ci);
                        u[0] = p.x; u[1] = p.y; u[2] = p.z; u[3] = p.w;
                    }
                    const float mu = warp_sum(sum4(u)) / (float)d;
#pragma unroll
                    for (int j = 0; j < 4; ++j) u[j] = ci + j < d ? u[j] - mu : 0.0f;
                    const float r = r_rsqrt(warp_sum(dot4(u, u)) / (float)d + a.eps);
#pragma unroll
                    for (int j = 0; j < 4; ++j) u[j] *= r;
                    if (key)
#pragma unroll
                        for (int j = 0; j < 4; ++j) x[j] = x[j] + u[j] - vv[j];
                    const float sx = warp_sum(sum4(x)) / (float)d, sxy = warp_sum(dot4(x, u)) / (float)d;
#pragma unroll
                    for (int j = 0; j < 4; ++j) out[j] = ci + j < d ? r * (x[j] - sx - u[j] * sxy) : 0.0f;
                    if (key && lane == 0) { sl[tl.sr + t] = r; sl[tl.smey + t] = sxy; }
                }
                if (ci < dp) {
                    st_split4<true>(blk(key ? tl.sPu : tl.sUq) + (size_t)(tk * db + (lane >> 4)) * B, t & 63, ci & 63, out);
                    if (key) {
                        *reinterpret_cast<float4*>(sl + tl.sy + (size_t)t * dp + ci) = make_float4(u[0], u[1], u[2], u[3]);
                        *reinterpret_cast<float4*>(sl + tl.spu + (size_t)t * dp + ci) = make_float4(out[0], out[1], out[2], out[3]);
                    }
                }
            }
        }
        G.sync_cta();

        // back through the last matrix: ph, pz (keys) and the adjoint of z (queries)
        for (int b0 = 0; b0 < hb; b0 += 2) {
            const bool two = b0 + 1 < hb;
            const unsigned char* pw = blk(tl.sW[LAST]) + (size_t)b0 * db * B;
            const Opnd x{blk(tl.sPu) + (size_t)tk * db * B, blk(tl.sUq) + (size_t)tk * db * B, B, true, false};
            const Opnd w[1] = {{pw, two ? pw + (size_t)db * B : nullptr, B, true, false}};
            G.job_begin();
            G.term<1>(db, false, x, w, {0u});
            G.job_end([&](uint32_t t) {
                const int bl = b0 + (row >> 6);
                const bool key = grp < 2;
#pragma unroll 1
                for (int half = 0; half < 2; ++half) {
                    const int col = 32 * grp + 16 * half, tok = col & 63;
                    float ph[16], cv[16];
                    acc16(t + col, ph);
                    if (row >= 64 && !two) continue;
                    const size_t e0 = (((size_t)bl * tb + tk) * 64 + tok) * 64 + (row & 63);
                    const size_t ho = ((size_t)bl * tb + tk) * B;
                    if (key) {
                        float* c4 = sl + tl.sc4 + e0;
#pragma unroll
                        for (int j = 0; j < 16; ++j) cv[j] = c4[64 * j];
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            c4[64 * j] = ph[j] * cv[j];
                            sl[tl.sph + e0 + 64 * j] = ph[j];
                        }
                    }
#pragma unroll
                    for (int i = 0; i < LAST; ++i) {
                        const float* cf = sl + (key ? (i ? tl.sc2 : tl.sc1) : (i ? tl.sc2q : tl.sc1q)) + e0;
#pragma unroll
                        for (int j = 0; j < 16; ++j) cv[j] = cf[64 * j];
#pragma unroll
                        for (int j = 0; j < 16; ++j) cv[j] *= ph[j];
                        st_split16(blk(key ? tl.sPz[i] : tl.sZq[i]) + ho, row & 63, tok, cv);
                    }
                }
            });
        }
        G.sync_cta();

        // dq = d_o + W_first^T zqb
        G.job_begin();
#pragma unroll
        for (int i = 0; i < LAST; ++i) {
            const unsigned char* pw = blk(tl.sW[i]);
            const Opnd z{blk(tl.sZq[i]) + (size_t)tk * B, nullptr, (uint32_t)tb * B, true, true};
            const Opnd w[1] = {{pw, db == 2 ? pw + B : nullptr, (uint32_t)db * B, true, false}};
            G.term<1>(hb, false, z, w, {0u});
        }
        G.job_end([&](uint32_t t) {
            const int tok = 16 * grp, n = min(16, len - tk * 64 - tok);
            float x[16], g[16];
            acc16(t + tok, x);
            const size_t e0 = (size_t)(tk * 64 + tok) * d + row;
#pragma unroll
            for (int j = 0; j < 16; ++j) g[j] = row < d && j < n ? __bfloat162float(doc[e0 + (size_t)j * d]) : 0.0f;
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (row < d && j < n) dqc[e0 + (size_t)j * d] = __float2bfloat16_rn(g[j] + x[j]);
        });
    }
    G.teardown();
}

}  // namespace tile
}  // namespace e2ttt
