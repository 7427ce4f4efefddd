// Block-tiled forward, chunks of several blocks of 64 tokens: one launch of persistent CTAs that take work items off a queue.
//
// A cluster per sequence (tile_fwd.cu) walks five phases per chunk, each ending in a barrier, and everything a phase leaves for the next -
// 20 MB per chunk of 512 tokens at d = 128, h = 512 - is stored by threads at 18-31 B/clk and SM and read back through L2 and HBM.  All tokens
// of a chunk see the same weights, so the chunk is cut twice instead (64 sequences of 4096 tokens: 2990 -> 1750 us):
//   tokens item  (sequence, chunk, 64 tokens)            z, activations, u, layer norm, outputs, pu.  All hidden units, 128 at a time: the
//                                                        activations go from tensor memory to a shared-memory tile that the second
//                                                        product reads; u never leaves tensor memory.  What is left for the other
//                                                        items: the keys' activations (bulk copies out of that tile), act'(z), pu.
//   weights item (sequence, chunk, matrix, 128 hidden)   pz (first matrices), both weighted aggregations over all tokens of the chunk in
//                                                        tensor memory, state transition, operand blocks of the next chunk's weights.
//   norm item    (post-chunk normalisation only)         rows of the new weights, their operand blocks.
// Items depend on earlier items of the same sequence: counters per sequence, waited for by the copy warp.  The queue hands items out in
// an order in which every item comes after those it depends on, so the earliest unfinished item can always run, however many CTAs there are.
// Sequences are taken in sets and, inside a set, out of step with each other: while one is at its tokens another is at its weights, and
// as many items lie between dependent ones as the GPU has in work (flow_plan, tile_flow.h).
//
// What bounds it now: a tokens item of 128 x 512 takes 79 thousand cycles, 46 of them on the activations - their instructions, half of it, and waits
// for products and for the tile between them - a weights item of 512 tokens 71 (first matrices) and 40 (last).  An SM stores 32 B/clk, threads or bulk
// copies alike, but 16 where a warp's lanes write 32 bytes of 32 lines (st_split16): tiles that are in shared memory anyway leave by bulk copies.
//
// 20 warps: 0-15 epilogues (warp w: lanes 32 (w & 3).., group w >> 2 of the columns), 16 copies operand blocks, 17 issues MMAs and the
// bulk stores of the tiles that it reads, 18 reports finished items.  setmaxnreg gives the epilogues the control warps' registers.
#include "tile.cuh"
#include "tile_flow.h"

namespace e2ttt {
using namespace tile;

namespace {

constexpr uint32_t B = 2 * kHalf;       // bytes of an operand block
constexpr int kFlowThreads = 640;
constexpr int kCells = 3, kAllCells = 7;  // ring of 32 KB; the last matrix' items, which need nothing else, stream through all of shared memory
constexpr uint32_t kCell = 32768;
// Shared memory: tile of activations (tokens) or of the scaled pz (weights) | tokens' rows (tokens) or the last matrix (weights) | ring
constexpr uint32_t kTileBytes = 65536, kSideBytes = 65536;
constexpr uint32_t kU = 256, kPh = 256;  // tensor-memory columns of u (two sums of 128) and of ph (two of 64); z and the aggregates: 0..255
// u is summed over 8 x 128 hidden units at a time: every MMA truncates the sum it adds to.  The sums are added in fp32, by the threads that will
// need them, in the workspace (where other kernels keep the queries' activations).  Error of the chunk-end states against 64 bits after two chunks of
// 64 tokens, d = 128, in one sum -> this way: h = 8192 8.9e-6 -> 4.9e-6, 3072 5.5e-6 -> 4.9e-6 (operands of two bf16 terms alone: 4.4e-6).  33
// sequences of two chunks, h = 2048: 376 -> 384 us.  Up to 1024 hidden units there is one sum, and the kernel is compiled without this
constexpr int kUSteps = 8;

struct FlowArgs {
    SimtFwdArgs a;
    FlowPlan p;
};

struct FlowShared {
    uint64_t full[kAllCells], empty[kAllCells];
    uint64_t written[2];                  // by the item's parity: all epilogue warps have stored its results
    uint64_t item[2], go[2], fin[2];      // by the item's parity: number known; what it depends on is done; finished
    uint64_t side_free, x_full, w_full;   // rows / last matrix: read by all MMAs, copies and warps of the item; written
    uint64_t tile_free;                   // tile: read by all MMAs, copies and warps of the item
    uint64_t acc_free;                    // tensor memory read out, once per item
    uint64_t z_full[2], z_empty[2], a_full, a_empty, u_full, stored;
    uint64_t ph_full[2], ph_empty[2], pz_full[2], pz_empty[2], acc_full;
    int4 id[2];               // the item: type, sequence, chunk, part
    int cur[2];               // what the epilogue warps agree on: the item stands (0 once a wait has given up)
    uint32_t tmem;
    int dead;
    float kb[16][32];  // per epilogue warp: K^W, then K^M, of its 16 tokens
};
constexpr size_t kFlowSmem = kTileBytes + kSideBytes + kCells * kCell + sizeof(FlowShared);
static_assert(kFlowSmem <= 232448, "227 KB of shared memory per CTA");

// Counters of a sequence, in its slice of the workspace; the queue is in sequence 0's
struct Counters {
    unsigned tokens, weights, norms, pad;
    unsigned long long queue;
};

// The order in which copy and MMA warps go through the cells, and the parity of a cell's next load
struct Cells {
    uint32_t bits = 0;
    int ring = 0, at = -1;  // next cell of the ring; place in the longer one, -1: not in use
    __device__ void all(bool on) { at = on ? 0 : -1; }
    __device__ uint32_t next() {  // the longer ring starts with the cells that are next in the shorter one
        const uint32_t u = at < 0 || at < kCells ? ring : at;
        if (at < kCells) ring = ring + 1 == kCells ? 0 : ring + 1;
        if (at >= 0) at = at + 1 == kAllCells ? 0 : at + 1;
        return u;
    }
    __device__ uint32_t parity(uint32_t u) const { return bits >> u & 1; }
    __device__ void used(uint32_t u) { bits ^= 1u << u; }
};

__device__ __forceinline__ void bulk_s2g(void* dst, uint32_t src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// 8 consecutive values of one row of a 64 x 64 block in shared memory (hi; lo `lo` bytes behind)
__device__ __forceinline__ void sts_split8(uint32_t blk, uint32_t lo, int row, int col0, const float (&v)[8]) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const __nv_bfloat162 hh = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
        const float2 hf = __bfloat1622float2(hh);
        h[j] = *reinterpret_cast<const uint32_t*>(&hh);
        l[j] = pack_bf16(v[2 * j] - hf.x, v[2 * j + 1] - hf.y);
    }
    const uint32_t at = blk + row * 128 + (((col0 >> 3) ^ (row & 7)) << 4);
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(at), "r"(h[0]), "r"(h[1]), "r"(h[2]), "r"(h[3]) : "memory");
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(at + lo), "r"(l[0]), "r"(l[1]), "r"(l[2]), "r"(l[3]) : "memory");
}
// 8 values of a token's row at column c, 0 beyond d
__device__ __forceinline__ uint4 ld_row8(const __nv_bfloat16* row, int c, int d) {
    if ((d & 7) == 0) return c < d ? *reinterpret_cast<const uint4*>(row + c) : make_uint4(0u, 0u, 0u, 0u);
    if ((d & 3) == 0) {  // rows of 8 bytes' alignment
        const uint2 x = c < d ? *reinterpret_cast<const uint2*>(row + c) : make_uint2(0u, 0u);
        const uint2 y = c + 4 < d ? *reinterpret_cast<const uint2*>(row + c + 4) : make_uint2(0u, 0u);
        return make_uint4(x.x, x.y, y.x, y.y);
    }
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t lo = c + 2 * j < d ? (uint32_t)__bfloat16_as_ushort(row[c + 2 * j]) : 0u;
        const uint32_t hi = c + 2 * j + 1 < d ? (uint32_t)__bfloat16_as_ushort(row[c + 2 * j + 1]) : 0u;
        w[j] = lo | hi << 16;
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ void unpack8(const uint4& r, float (&v)[8]) {
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        v[2 * j] = __uint_as_float(w[j] << 16);
        v[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
    }
}

// WIDE: more than kUSteps slices of 128 hidden units
template <int KIND, bool WIDE> __global__ void __launch_bounds__(kFlowThreads, 1) tile_flow_kernel(const FlowArgs f) {
    constexpr int NMAT = (KIND == 0) ? 2 : 3, LAST = NMAT - 1;
    constexpr bool SW = KIND == 1;
    constexpr uint32_t NZ = SW ? 1 : 2;  // accumulators of z
    extern __shared__ __align__(1024) unsigned char flow_smem[];
    const SimtFwdArgs& a = f.a;
    const uint32_t tile0 = smem_u32(flow_smem), side0 = tile0 + kTileBytes, ring0 = side0 + kSideBytes;
    FlowShared& sh = *reinterpret_cast<FlowShared*>(flow_smem + kTileBytes + kSideBytes + kCells * kCell);
    // (from lane 0: the compiler then knows that it is the same for the warp, and keeps what follows from it in uniform registers)
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kAllCells; ++i) { mbar_init(&sh.full[i], 1); mbar_init(&sh.empty[i], 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh.item[i], 1); mbar_init(&sh.go[i], 1); mbar_init(&sh.fin[i], 1); mbar_init(&sh.written[i], 16);
            mbar_init(&sh.z_full[i], 1); mbar_init(&sh.z_empty[i], 16);
            mbar_init(&sh.ph_full[i], 1); mbar_init(&sh.ph_empty[i], 16);
            mbar_init(&sh.pz_full[i], 16); mbar_init(&sh.pz_empty[i], 1);
        }
        mbar_init(&sh.side_free, 18); mbar_init(&sh.x_full, 16); mbar_init(&sh.w_full, 1); mbar_init(&sh.acc_free, 16); mbar_init(&sh.tile_free, 16);
        mbar_init(&sh.a_full, 16); mbar_init(&sh.a_empty, 2); mbar_init(&sh.u_full, 1); mbar_init(&sh.stored, 1); mbar_init(&sh.acc_full, 1);
        sh.dead = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(&sh.tmem, 512);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = __shfl_sync(0xffffffffu, sh.tmem, 0);
    WaitCtx wc;
    wc.dead = &sh.dead;
    wc.status = a.status;

    const SimtLayout& lay = a.lay;
    const TileLayout& tl = lay.tl;
    const int d = a.d, h = a.h, db = tl.db, hb = tl.hb, tb = tl.tb, dp = db * 64, ns = f.p.ns;
    const size_t dh = (size_t)d * h;
    const bool normed = a.row_norm[0] != nullptr, queries = a.o != nullptr;
    auto ws_of = [&](int seq) { return reinterpret_cast<float*>(a.ws) + (size_t)seq * lay.per_seq; };
    auto counters = [&](int seq) { return reinterpret_cast<Counters*>(ws_of(seq) + tl.fred); };
    // the last matrix' blocks in two buffers by the chunk's parity: its weights item writes the next ones while others read these
    auto wb_of = [&](int i, int c) { return i == LAST && (c & 1) ? tl.fPzW[0] : tl.Wb[i]; };
    auto tokens_of = [&](int c) { return min(a.C, a.L - c * a.C); };
    auto await = [&](uint64_t* bar, uint32_t use, int where) {
        mbar_wait(bar, use & 1, wc, where);
        tc_fence_after_sync();
    };
    auto item_of = [&](uint32_t n) {
        const int4 x = sh.id[n & 1];
        return FlowItem{__shfl_sync(0xffffffffu, x.x, 0), __shfl_sync(0xffffffffu, x.y, 0), __shfl_sync(0xffffffffu, x.z, 0), __shfl_sync(0xffffffffu, x.w, 0)};
    };
    auto cell_at = [&](uint32_t u) { return u < kCells ? ring0 + u * kCell : tile0 + (u - kCells) * kCell; };
    auto given_up = [&] { return __any_sync(0xffffffffu, *wc.dead != 0); };
    auto arrive1 = [&](uint64_t* bar) {
        __syncwarp();
        if (lane == 0) mbar_arrive(bar);
    };

    if (warp >= kEpiWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    if (warp == kEpiWarps) {
        // ================================================================= copy warp
        Cells cells;
        auto cell_begin = [&](uint32_t bytes) {
            const uint32_t u = cells.next();
            mbar_wait(&sh.empty[u], cells.parity(u) ^ 1, wc, 501);
            cells.used(u);
            if (lane == 0) mbar_expect_tx(&sh.full[u], bytes);
            return u;
        };
        auto load = [&](const unsigned char* p0, const unsigned char* p1) {  // one or two blocks: hi, hi | lo, lo
            const uint32_t u = cell_begin(kHalf * (p1 ? 4 : 2)), dst = cell_at(u);
            if (lane == 0) {
                for (int part = 0; part < 2; ++part) {
                    bulk_g2s(dst + part * B, p0 + part * kHalf, kHalf, &sh.full[u]);
                    if (p1) bulk_g2s(dst + part * B + kHalf, p1 + part * kHalf, kHalf, &sh.full[u]);
                }
            }
            __syncwarp();
        };
        auto load_flat = [&](const unsigned char* p, uint32_t bytes) {
            const uint32_t u = cell_begin(bytes);
            if (lane == 0)
                for (uint32_t at = 0; at < bytes; at += kHalf) bulk_g2s(cell_at(u) + at, p + at, kHalf, &sh.full[u]);
            __syncwarp();
        };
        unsigned long long* queue = &counters(0)->queue;
        for (uint32_t n = 0;; ++n) {
            if (n >= 2) mbar_wait(&sh.fin[n & 1], ((n >> 1) - 1) & 1, wc, 502);
            FlowItem it;
            do {
                unsigned long long x = 0;
                if (lane == 0) x = atomicAdd(queue, 1ull);
                it = flow_item(f.p, (long long)__shfl_sync(0xffffffffu, x, 0));
            } while (it.type == kFlowNone);
            if (lane == 0) sh.id[n & 1] = make_int4(it.type, it.seq, it.c, it.part);
            arrive1(&sh.item[n & 1]);
            if (it.type == kFlowEnd || given_up()) break;
            const int c = it.c, tbn = (tokens_of(c) + 63) / 64;
            float* ws = ws_of(it.seq);
            auto blk = [&](size_t off) { return reinterpret_cast<const unsigned char*>(ws + off); };
            {   // what the item depends on
                const Counters* cn = counters(it.seq);
                const unsigned* p = it.type == kFlowTokens ? (normed ? &cn->norms : &cn->weights) : it.type == kFlowWeights ? &cn->tokens : &cn->weights;
                const unsigned need = it.type == kFlowTokens ? (unsigned)c * (normed ? f.p.n3 : f.p.n2)
                                      : it.type == kFlowWeights ? (unsigned)(c * tb + tbn) : (unsigned)(c + 1) * f.p.n2;
                if (need && ld_acquire(p) < need && !*wc.dead) {
                    const long long t0 = clock64();
                    while (ld_acquire(p) < need) {
                        __nanosleep(40);
                        if (*wc.dead) break;
                        if (clock64() - t0 > wc.limit) {
                            *wc.dead = 1;
                            atomicCAS(wc.status, 0, 503);
                            break;
                        }
                    }
                }
                __syncwarp();
                fence_proxy_async_all();
                arrive1(&sh.go[n & 1]);
            }
            if (it.type == kFlowTokens) {
                const unsigned char* wl = blk(wb_of(LAST, c));
                for (int b = 0; b <= ns; ++b) {
                    if (b < ns)
                        for (int k = 0; k < db; ++k)
#pragma unroll
                            for (int i = 0; i < LAST; ++i) {
                                const unsigned char* p = blk(tl.Wb[i]) + ((size_t)2 * b * db + k) * B;
                                load(p, 2 * b + 1 < hb ? p + (size_t)db * B : nullptr);
                            }
                    if (b > 0)
                        for (int j = 2 * b - 2; j < min(hb, 2 * b); ++j) {
                            const unsigned char* p = wl + (size_t)j * db * B;
                            load(p, db == 2 ? p + B : nullptr);
                        }
                }
            } else if (it.type == kFlowWeights) {
                const int i = it.part / ns, b0 = 2 * (it.part % ns);
                const bool two = b0 + 1 < hb;
                if (i < LAST) {
                    if (n >= 1) mbar_wait(&sh.side_free, (n - 1) & 1, wc, 504);
                    fence_proxy_async_smem();
                    if (lane == 0) {
                        mbar_expect_tx(&sh.w_full, (uint32_t)db * B * (two ? 2u : 1u));
                        for (int k = 0; k < db; ++k)
                            for (int j = 0; j < (two ? 2 : 1); ++j)
                                for (int part = 0; part < 2; ++part)
                                    bulk_g2s(side0 + k * kCell + part * B + j * kHalf, blk(wb_of(LAST, c)) + ((size_t)(b0 + j) * db + k) * B + part * kHalf, kHalf, &sh.w_full);
                    }
                    __syncwarp();
                    for (int tk = 0; tk <= tbn; ++tk) {
                        if (tk < tbn) load_flat(blk(tl.fPu) + (size_t)tk * db * B, db * B);
                        if (tk > 0) load_flat(blk(tl.fK[0]) + (size_t)(tk - 1) * db * kHalf, db * kHalf);
                    }
                } else {
                    cells.all(true);
                    for (int tk = 0; tk < tbn; ++tk) {
                        if (n >= 1 && tk == 1) {  // from the fourth cell on
                            mbar_wait(&sh.side_free, (n - 1) & 1, wc, 505);
                            mbar_wait(&sh.tile_free, (n - 1) & 1, wc, 506);
                            fence_proxy_async_smem();
                        }
                        const unsigned char* p = blk(tl.fA) + ((size_t)b0 * tb + tk) * B;
                        load(p, two ? p + (size_t)tb * B : nullptr);
                        load_flat(blk(tl.fPuW) + (size_t)tk * db * B, db * B);
                        load_flat(blk(tl.fPuM) + (size_t)tk * db * B, db * B);
                    }
                    cells.all(false);
                }
            }
        }
    } else if (warp == kEpiWarps + 1) {
        // ================================================================= MMA warp
        const bool issue = lane == 0;
        Cells cells;
        uint32_t nx = 0, nw = 0, nz = 0, na = 0, nph = 0, npz = 0;
        auto take = [&](uint32_t& u) {
            u = cells.next();
            await(&sh.full[u], cells.parity(u), 511);
            cells.used(u);
            return cell_at(u);
        };
        for (uint32_t n = 0;; ++n) {
            await(&sh.item[n & 1], n >> 1, 512);
            const FlowItem it = item_of(n);
            if (it.type == kFlowEnd || given_up()) break;
            if (n >= 1) await(&sh.acc_free, n - 1, 513);
            const int c = it.c, tbn = (tokens_of(c) + 63) / 64;
            float* ws = ws_of(it.seq);
            auto blk = [&](size_t off) { return reinterpret_cast<unsigned char*>(ws + off); };
            if (it.type == kFlowTokens) {
                const int tk = it.part;
                await(&sh.x_full, nx++, 514);
                await(&sh.go[n & 1], n >> 1, 535);  // the chunk before has been read
                if (issue) {  // the keys' rows, for the weights items
                    for (int k = 0; k < db; ++k) bulk_s2g(blk(tl.fK[0]) + ((size_t)tk * db + k) * kHalf, side0 + k * B, kHalf);
                    bulk_commit();
                }
                __syncwarp();
                for (int b = 0; b <= ns; ++b) {
                    if (b < ns) {
                        const uint32_t set = nz % NZ, idesc = make_idesc(128, queries ? 128 : 64, true, false);
                        if (nz >= NZ) await(&sh.z_empty[set], nz / NZ - 1, 515);
#pragma unroll 1
                        for (int k = 0; k < db; ++k)
#pragma unroll
                            for (int i = 0; i < LAST; ++i) {
                                uint32_t u;
                                const uint32_t w = take(u), dst = tmem + set * 128 + i * 128;
                                const uint64_t w0 = make_smem_desc(w, kHalf, 1024), x0 = make_smem_desc(side0 + k * B, kHalf, 1024);
#pragma unroll
                                for (int ks = 0; ks < 4; ++ks) {
                                    const uint64_t wh = w0 + ks * (2048 >> 4), xd = x0 + ks * (32 >> 4);
                                    umma_bf16_elect(dst, wh + (B >> 4), xd, idesc, k > 0 || ks > 0, issue);
                                    umma_bf16_elect(dst, wh, xd, idesc, true, issue);
                                }
                                umma_commit_elect(&sh.empty[u], issue);
                            }
                        umma_commit_elect(&sh.z_full[set], issue);
                        if (b == ns - 1) umma_commit_elect(&sh.side_free, issue);
                        ++nz;
                    }
                    if (b > 0) {
                        const int b0 = 2 * b - 2, nj = min(hb - b0, 2);
                        await(&sh.a_full, na++, 516);
                        if (issue) {  // the keys' activations, for the last matrix' weights items
                            for (int j = 0; j < nj; ++j)
                                for (int part = 0; part < 2; ++part)
                                    bulk_s2g(blk(tl.fA) + ((size_t)(b0 + j) * tb + tk) * B + part * kHalf, tile0 + j * kCell + part * B, kHalf);
                            bulk_commit();
                        }
                        __syncwarp();
                        const uint32_t idesc = make_idesc(128, db == 2 ? 128 : 64, true, true);
#pragma unroll 1
                        for (int j = 0; j < nj; ++j) {
                            uint32_t u;
                            const uint32_t w = take(u);
                            const uint64_t a0 = make_smem_desc(tile0 + j * kCell, kHalf, 1024), w0 = make_smem_desc(w, kHalf, 1024);
#pragma unroll
                            for (int ks = 0; ks < 4; ++ks) {
                                const uint64_t ah = a0 + ks * (2048 >> 4), wh = w0 + ks * (2048 >> 4);
                                const bool acc = (WIDE ? (b - 1) % kUSteps != 0 : b > 1) || j > 0 || ks > 0;
                                // the small terms in a sum of their own: every MMA truncates the sum it adds to
                                umma_bf16_elect(tmem + kU + 128, ah + (B >> 4), wh, idesc, acc, issue);
                                umma_bf16_elect(tmem + kU + 128, ah, wh + (B >> 4), idesc, true, issue);
                                umma_bf16_elect(tmem + kU, ah, wh, idesc, acc, issue);
                            }
                            umma_commit_elect(&sh.empty[u], issue);
                        }
                        umma_commit_elect(&sh.a_empty, issue);
                        if (b == ns || (WIDE && b % kUSteps == 0)) umma_commit_elect(&sh.u_full, issue);
                        if (issue) {
                            bulk_wait_read();
                            mbar_arrive(&sh.a_empty);
                            if (b == 1) mbar_arrive(&sh.side_free);
                        }
                        __syncwarp();
                    }
                }
                if (issue) {
                    bulk_wait();
                    fence_proxy_async_all();
                    mbar_arrive(&sh.stored);
                }
                __syncwarp();
            } else if (it.type == kFlowWeights && it.part / ns < LAST) {
                const int b0 = 2 * (it.part % ns);
                const bool two = b0 + 1 < hb;
                await(&sh.w_full, nw++, 517);
                const uint32_t idp = make_idesc(128, 64, false, false), ida = make_idesc(128, two ? 128 : 64, true, false);
#pragma unroll 1
                for (int tk = 0; tk <= tbn; ++tk) {
                    if (tk < tbn) {  // ph = W_last^T pu: hidden units on the lanes
                        const uint32_t set = nph & 1;
                        if (nph >= 2) await(&sh.ph_empty[set], (nph >> 1) - 1, 518);
                        uint32_t u;
                        const uint32_t p = take(u), dst = tmem + kPh + set * 64;
#pragma unroll 1
                        for (int k = 0; k < db; ++k) {
                            const uint64_t w0 = make_smem_desc(side0 + k * kCell, kHalf, 1024), p0 = make_smem_desc(p + k * B, kHalf, 1024);
#pragma unroll
                            for (int ks = 0; ks < 4; ++ks) {
                                const uint64_t wh = w0 + ks * (32 >> 4), ph = p0 + ks * (32 >> 4);
                                umma_bf16_elect(dst, wh + (B >> 4), ph, idp, k > 0 || ks > 0, issue);
                                umma_bf16_elect(dst, wh, ph + (kHalf >> 4), idp, true, issue);
                                umma_bf16_elect(dst, wh, ph, idp, true, issue);
                            }
                        }
                        umma_commit_elect(&sh.empty[u], issue);
                        umma_commit_elect(&sh.ph_full[set], issue);
                        if (tk == tbn - 1) umma_commit_elect(&sh.side_free, issue);
                        ++nph;
                    }
                    if (tk > 0) {  // both aggregations of 64 tokens: d on the lanes
                        uint32_t u;
                        const uint32_t kt = take(u);
#pragma unroll 1
                        for (int m = 0; m < 2; ++m) {
                            await(&sh.pz_full[m], npz, 519);
                            const uint64_t k0 = make_smem_desc(kt, kHalf, 1024), z0 = make_smem_desc(tile0 + m * kCell, kHalf, 1024);
#pragma unroll
                            for (int ks = 0; ks < 4; ++ks) {
                                const uint64_t kd = k0 + ks * (2048 >> 4), zh = z0 + ks * (32 >> 4);
                                umma_bf16_elect(tmem + m * 128, kd, zh + (B >> 4), ida, tk > 1 || ks > 0, issue);
                                umma_bf16_elect(tmem + m * 128, kd, zh, ida, true, issue);
                            }
                            umma_commit_elect(&sh.pz_empty[m], issue);
                        }
                        ++npz;
                        umma_commit_elect(&sh.empty[u], issue);
                    }
                }
                arrive1(&sh.side_free);
                umma_commit_elect(&sh.acc_full, issue);
            } else if (it.type == kFlowWeights) {
                const uint32_t ida = make_idesc(128, db == 2 ? 128 : 64, false, true);
                cells.all(true);
#pragma unroll 1
                for (int tk = 0; tk < tbn; ++tk) {  // hidden units on the lanes
                    uint32_t ua, up;
                    const uint32_t at = take(ua);
#pragma unroll 1
                    for (int m = 0; m < 2; ++m) {
                        const uint32_t p = take(up);
                        const uint64_t a0 = make_smem_desc(at, kHalf, 1024), p0 = make_smem_desc(p, B, 1024);
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) {
                            const uint64_t ah = a0 + ks * (32 >> 4), ph = p0 + ks * (2048 >> 4);
                            umma_bf16_elect(tmem + m * 128, ah + (B >> 4), ph, ida, tk > 0 || ks > 0, issue);
                            umma_bf16_elect(tmem + m * 128, ah, ph + (kHalf >> 4), ida, true, issue);
                            umma_bf16_elect(tmem + m * 128, ah, ph, ida, true, issue);
                        }
                        umma_commit_elect(&sh.empty[up], issue);
                    }
                    umma_commit_elect(&sh.empty[ua], issue);
                }
                cells.all(false);
                umma_commit_elect(&sh.side_free, issue);
                arrive1(&sh.side_free);
                umma_commit_elect(&sh.acc_full, issue);
            } else {
                if (issue) { mbar_arrive(&sh.side_free); mbar_arrive(&sh.side_free); }
                __syncwarp();
            }
        }
    } else if (warp == kEpiWarps + 2) {
        // ================================================================= reports: what threads wrote is read by other CTAs, by loads
        // and by bulk copies.  A warp of its own: the fence waits for all of the item's stores
        for (uint32_t n = 0;; ++n) {
            mbar_wait(&sh.item[n & 1], (n >> 1) & 1, wc, 541);
            const FlowItem it = item_of(n);
            if (it.type == kFlowEnd || given_up()) break;
            mbar_wait(&sh.written[n & 1], (n >> 1) & 1, wc, 542);
            if (lane == 0) {
                Counters* cn = counters(it.seq);
                __threadfence();
                atomicAdd(it.type == kFlowTokens ? &cn->tokens : it.type == kFlowWeights ? &cn->weights : &cn->norms, 1u);
            }
            arrive1(&sh.fin[n & 1]);
        }
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
        // ================================================================= epilogue warps
        const int q4 = warp & 3, grp = warp >> 2, row = 32 * q4 + lane;
        const uint32_t lanes = tmem + ((uint32_t)(32 * q4) << 16);
        auto epi_sync = [] { asm volatile("bar.sync 1, 512;" ::: "memory"); };
        auto signal = [&](uint64_t* bar) {  // this warp's part of a tile in shared memory is written (a fence of global memory as
            fence_proxy_async_smem();       // well would wait for the stores under way: 2 us of every item)
            arrive1(bar);
        };
        auto release = [&](uint64_t* bar) {  // this warp has read its part of tensor memory
            tc_fence_before_sync();
            arrive1(bar);
        };
        // parities of the waits, a bit each (registers are short: a spilled value comes from L2)
        enum { kZ = 1, kA = 4, kUB = 8, kP = 16, kPz = 64, kAcc = 128, kSt = 256 };  // kZ, kP: two bits, accumulator and parity
        uint32_t par = 0;
        auto bit = [&](uint32_t b) { return (par & b) != 0 ? 1u : 0u; };
        for (uint32_t n = 0;; ++n) {
            if (warp == 0) {  // the item's barriers below are for all of these warps or none
                await(&sh.item[n & 1], n >> 1, 521);
                if (lane == 0) sh.cur[n & 1] = *wc.dead == 0;
            }
            epi_sync();
            if (!sh.cur[n & 1]) break;
            const FlowItem it = item_of(n);
            if (it.type == kFlowEnd) break;
            const int c = it.c, seq = it.seq, s = c * a.C, len = tokens_of(c), tbn = (len + 63) / 64;
            const bool last_chunk = c + 1 == a.nchunks;
            float* ws = ws_of(seq);
            auto blk = [&](size_t off) { return reinterpret_cast<unsigned char*>(ws + off); };
            ChunkScalars<float>* scs = reinterpret_cast<ChunkScalars<float>*>(ws + tl.fslot);
            const ChunkScalars<float>& sc = scs[c & 1];
            const size_t tok0 = ((size_t)seq * a.Ls + s) * d;
            auto u_sum = [&](int tk, int i) { return ws + tl.fAq + ((size_t)(tk * 4 + i) * 512 + threadIdx.x) * 8; };  // 8 of this thread's 32 columns
            if (it.type == kFlowTokens) {
                const int tk = it.part;
                // ---- rows of the keys (0-63) and queries (64-127) -> operand slabs
                if (n >= 1) await(&sh.side_free, n - 1, 522);
                {
                    const int rr = threadIdx.x >> 2, part = threadIdx.x & 3, t = tk * 64 + (rr & 63);
                    const __nv_bfloat16* src = reinterpret_cast<const __nv_bfloat16*>(rr < 64 ? a.k : a.q) + tok0 + (size_t)t * d;
                    uint4 x[4];
                    auto put = [&](uint32_t at) {
                        if (32 * part < dp)
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(at + ((((part & 1) * 4 + i) ^ (rr & 7)) << 4)), "r"(x[i].x),
                                             "r"(x[i].y), "r"(x[i].z), "r"(x[i].w)
                                             : "memory");
                    };
#pragma unroll
                    for (int i = 0; i < 4; ++i) x[i] = t < len ? ld_row8(src, 32 * part + 8 * i, d) : make_uint4(0u, 0u, 0u, 0u);
                    put(side0 + (part >> 1) * B + rr * 128);
                    if (rr < 64) {  // the values, for the layer norm's rows
                        src = reinterpret_cast<const __nv_bfloat16*>(a.v) + tok0 + (size_t)t * d;
#pragma unroll
                        for (int i = 0; i < 4; ++i) x[i] = t < len ? ld_row8(src, 32 * part + 8 * i, d) : make_uint4(0u, 0u, 0u, 0u);
                        put(side0 + 2 * B + (part >> 1) * kHalf + rr * 128);
                    }
                    signal(&sh.x_full);
                }
                await(&sh.go[n & 1], n >> 1, 523);
                // ---- a = act(z), 128 hidden units at a time
#pragma unroll 1
                for (int b = 0; b < ns; ++b) {
                    const int bl = 2 * b + (row >> 6);
                    const bool live = bl < hb;
                    const uint32_t set = SW ? 0u : bit(kZ), t = lanes + set * 128;
                    await(&sh.z_full[set], SW ? bit(kZ) : bit(2 * kZ), 524);
                    par ^= bit(kZ) ? 3 * kZ : kZ;
#pragma unroll 1
                    for (int half = 0; half < (queries ? 2 : 1); ++half) {
                        const bool key = half == 0;
#pragma unroll 1
                        for (int e = 0; e < 2; ++e) {
                            const uint32_t col = 64 * half + 16 * grp + 8 * e;
                            float z1[8], z2[8], act[8];
                            acc8(t + col, z1);
                            if (SW) acc8(t + 128 + col, z2);
                            if (e == 1 && half == (queries ? 1 : 0)) release(&sh.z_empty[set]);
                            if (key) {
                                float c1[8], c2[8];
#pragma unroll
                                for (int j = 0; j < 8; ++j) {
                                    if (!SW) {
                                        float cdf, pdf;
                                        normal_dist(z1[j], cdf, pdf);
                                        act[j] = z1[j] * cdf;
                                        c1[j] = cdf + z1[j] * pdf;
                                    } else {
                                        const float sg = sigmoid_hw(z1[j]), sl = z1[j] * sg;
                                        act[j] = sl * z2[j];
                                        c1[j] = z2[j] * (sg * (1.0f + z1[j] * (1.0f - sg)));
                                        c2[j] = sl;
                                    }
                                }
                                if (live) {
                                    const size_t e0 = ((size_t)bl * tb + it.part) * 4096 + (grp * 64 + (row & 63)) * 16 + 8 * e;
                                    st_f8(ws + tl.fc1 + e0, c1);
                                    if (SW) st_f8(ws + tl.fc2 + e0, c2);
                                }
                                if (e == 0 && b > 0) await(&sh.a_empty, bit(kA) ^ 1, 525);
                            } else {
#pragma unroll
                                for (int j = 0; j < 8; ++j) {
                                    if (!SW) {
                                        float cdf, pdf;
                                        normal_dist(z1[j], cdf, pdf);
                                        act[j] = z1[j] * cdf;
                                    } else {
                                        act[j] = z1[j] * sigmoid_hw(z1[j]) * z2[j];
                                    }
                                }
                            }
                            if (live) sts_split8(tile0 + (row >> 6) * kCell + (key ? 0u : kHalf), B, row & 63, 16 * grp + 8 * e, act);
                        }
                    }
                    par ^= kA;
                    if (WIDE && b > 0 && b % kUSteps == 0) {  // the MMAs that start the next sum wait for a_full
                        await(&sh.u_full, bit(kUB), 536);
                        par ^= kUB;
                        if (32 * grp < dp)
#pragma unroll 1
                            for (int i = 0; i < 4; ++i) {
                                float x[8], y[8];
                                acc8(lanes + kU + 32 * grp + 8 * i, x);
                                acc8(lanes + kU + 128 + 32 * grp + 8 * i, y);
#pragma unroll
                                for (int j = 0; j < 8; ++j) x[j] += y[j];
                                if (b > kUSteps) {
                                    ld_f8(u_sum(it.part, i), y);
#pragma unroll
                                    for (int j = 0; j < 8; ++j) x[j] += y[j];
                                }
                                st_f8(u_sum(it.part, i), x);
                            }
                        tc_fence_before_sync();
                    }
                    signal(&sh.a_full);
                }
                // ---- rows: token `row` (keys 0-63, queries 64-127), 32 columns; sums over the four groups of warps through what the
                // tile held of the queries' activations
                const bool key = row < 64;
                const int t = tk * 64 + (row & 63), c0 = 32 * grp;
                const bool live = t < len && (key || queries);
                const unsigned char* xs = flow_smem + kTileBytes + (c0 >> 6) * B + row * 128;  // this token's row, and its values
                const unsigned char* vs = flow_smem + kTileBytes + 2 * B + (c0 >> 6) * kHalf + (row & 63) * 128;
                const float kw = key && live ? sc.kW[t] : 0.0f, km = key && live ? sc.kM[t] : 0.0f;
                float u[32];
                await(&sh.u_full, bit(kUB), 526);
                par ^= kUB;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    float x[16], y[16];
                    acc16(lanes + kU + c0 + 16 * i, x);
                    acc16(lanes + kU + 128 + c0 + 16 * i, y);
#pragma unroll
                    for (int j = 0; j < 16; ++j) u[16 * i + j] = live && c0 + 16 * i + j < d ? x[j] + y[j] : 0.0f;
                }
                release(&sh.acc_free);
                if (WIDE && c0 < dp)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float y[8];
                        ld_f8(u_sum(tk, i), y);
#pragma unroll
                        for (int j = 0; j < 8; ++j) u[8 * i + j] += c0 + 8 * i + j < d ? y[j] : 0.0f;  // (nothing of a row past the end is used)
                    }
                float* red = reinterpret_cast<float*>(flow_smem + kHalf) + row;
                auto total = [&](int which, float x) {  // over the groups, in their order
                    red[which * 512 + grp * 128] = x;
                    epi_sync();
                    const float* p = red + which * 512;
                    return (p[0] + p[128]) + (p[256] + p[384]);
                };
                float x = 0.0f, y = 0.0f;
#pragma unroll
                for (int j = 0; j < 32; ++j) x += u[j];
                const float mu = total(0, x) / (float)d;
                x = 0.0f;
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    u[j] = c0 + j < d ? u[j] - mu : 0.0f;
                    x += u[j] * u[j];
                }
                const float r = r_rsqrt(total(1, x) / (float)d + a.eps);
                x = 0.0f;
                auto error = [&](int i, float (&e)[8]) {  // k + y - v, of 8 columns; of a query: its output
                    float vv[8];
                    const int at = ((((c0 >> 3) + i) ^ row) & 7) * 16;
                    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
                    unpack8(c0 < dp ? *reinterpret_cast<const uint4*>(xs + at) : zero, e);
                    unpack8(c0 < dp && key ? *reinterpret_cast<const uint4*>(vs + at) : zero, vv);
#pragma unroll
                    for (int j = 0; j < 8; ++j) e[j] = e[j] + u[8 * i + j] - vv[j];
                };
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float e[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) u[8 * i + j] *= r;
                    error(i, e);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        x += e[j];
                        y += e[j] * u[8 * i + j];
                    }
                }
                red[3 * 512 + grp * 128] = y;
                const float se = total(2, x) / (float)d;
                const float* py = red + 3 * 512;
                const float sey = ((py[0] + py[128]) + (py[256] + py[384])) / (float)d;
                if (key) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float e[8];
                        error(i, e);
#pragma unroll
                        for (int j = 0; j < 8; ++j) u[8 * i + j] = live && c0 + 8 * i + j < d ? r * (e[j] - se - u[8 * i + j] * sey) : 0.0f;
                    }
                    if (c0 < dp) {
                        const size_t off = (size_t)(tk * db + (c0 >> 6)) * B;
#pragma unroll 1
                        for (int which = 0; which < 3; ++which) {
                            const float k0 = which == 0 ? 1.0f : which == 1 ? kw : km;
                            unsigned char* to = blk(which == 0 ? tl.fPu : which == 1 ? tl.fPuW : tl.fPuM) + off;
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                float w[16];
#pragma unroll
                                for (int j = 0; j < 16; ++j) w[j] = k0 * u[16 * i + j];
                                st_split16(to, row & 63, (c0 & 63) + 16 * i, w);
                            }
                        }
                    }
                } else if (live) {
                    __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(a.o) + tok0 + (size_t)t * d;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float e[8];
                        error(i, e);
                        if ((d & 7) == 0) {
                            if (c0 + 8 * i < d)
                                *reinterpret_cast<uint4*>(o + c0 + 8 * i) = make_uint4(pack_bf16(e[0], e[1]), pack_bf16(e[2], e[3]), pack_bf16(e[4], e[5]), pack_bf16(e[6], e[7]));
                        } else if ((d & 3) == 0) {
#pragma unroll
                            for (int j = 0; j < 8; j += 4)
                                if (c0 + 8 * i + j < d)
                                    *reinterpret_cast<uint2*>(o + c0 + 8 * i + j) = make_uint2(pack_bf16(e[j], e[j + 1]), pack_bf16(e[j + 2], e[j + 3]));
                        } else {
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                if (c0 + 8 * i + j < d) o[c0 + 8 * i + j] = __float2bfloat16_rn(e[j]);
                        }
                    }
                }
                arrive1(&sh.side_free);
                await(&sh.stored, bit(kSt), 527);
                par ^= kSt;
                arrive1(&sh.tile_free);
            } else if (it.type == kFlowWeights) {
                const int i = it.part / ns, b0 = 2 * (it.part % ns);
                const bool two = b0 + 1 < hb;
                await(&sh.go[n & 1], n >> 1, 528);
                arrive1(&sh.side_free);
                if (it.part == 0 && warp == 15 && !last_chunk) {  // Algorithm 1 line 2 for the next chunk
                    const size_t t = (size_t)seq * a.Ls + s + a.C;
                    chunk_scalars_warp<float>(a.eta + t, a.beta + t, a.gamma + t, tokens_of(c + 1), &scs[(c + 1) & 1]);
                }
                if (i < LAST) {
                    const int bl = b0 + (row >> 6);
                    const bool live = bl < hb;
                    const float* cf = ws + (i == 0 ? tl.fc1 : tl.fc2) + (size_t)(live ? bl : b0) * tb * 4096 + (grp * 64 + (row & 63)) * 16;
                    float cv[2][8];
                    ld_f8(cf, cv[0]);
                    ld_f8(cf + 8, cv[1]);
                    float* kb = sh.kb[warp];
                    const float* kx = (lane < 16 ? sc.kW : sc.kM) + 16 * grp + (lane & 15);
                    auto ld_k = [&](int tk) { return tk * 64 + 16 * grp + (lane & 15) < len ? kx[tk * 64] : 0.0f; };
                    float kn = ld_k(0);
#pragma unroll 1
                    for (int tk = 0; tk < tbn; ++tk) {
                        const uint32_t set = bit(kP);
                        __syncwarp();
                        kb[lane] = kn;
                        __syncwarp();
                        if (tk + 1 < tbn) kn = ld_k(tk + 1);
                        await(&sh.ph_full[set], bit(2 * kP), 529);
                        par ^= set ? 3 * kP : kP;
                        float p[16];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            float x[8];
                            acc8(lanes + kPh + set * 64 + 16 * grp + 8 * e, x);
#pragma unroll
                            for (int j = 0; j < 8; ++j) p[8 * e + j] = x[j] * cv[e][j];
                        }
                        release(&sh.ph_empty[set]);
                        if (tk + 1 < tbn) {
                            ld_f8(cf + (size_t)(tk + 1) * 4096, cv[0]);
                            ld_f8(cf + (size_t)(tk + 1) * 4096 + 8, cv[1]);
                        }
#pragma unroll 1
                        for (int m = 0; m < 2; ++m) {
                            if (tk > 0) await(&sh.pz_empty[m], bit(kPz) ^ 1, 530);
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                float x[8];
#pragma unroll
                                for (int j = 0; j < 8; ++j) x[j] = kb[16 * m + 8 * e + j] * p[8 * e + j];
                                if (live) sts_split8(tile0 + m * kCell + (row >> 6) * kHalf, B, row & 63, 16 * grp + 8 * e, x);
                            }
                            signal(&sh.pz_full[m]);
                        }
                        par ^= kPz;
                    }
                }
                // ---- Algorithm 1 lines 4-7: the state transition
                const float cw = sc.cw, cm = sc.cm, cb = sc.cb;
                const float *w_in, *m_in;
                if (c == 0) {
                    const float* ck = a.init_slot >= 0 ? ws + lay.cck + (size_t)a.init_slot * 2 * NMAT * dh : nullptr;
                    w_in = ck ? ck + (size_t)i * dh : a.W_init[i] + (size_t)seq * dh;
                    m_in = ck ? ck + (size_t)(NMAT + i) * dh : (a.M_init[i] ? a.M_init[i] + (size_t)seq * dh : nullptr);
                } else if (a.save_states == 1) {
                    const float* ck = ws + lay.ckpt + (size_t)c * 2 * NMAT * dh;
                    w_in = ck + (size_t)i * dh; m_in = ck + (size_t)(NMAT + i) * dh;
                } else {
                    w_in = ws + lay.W[i]; m_in = ws + lay.M[i];
                }
                float *w_out = ws + lay.W[i], *m_out = ws + lay.M[i], *w_copy = nullptr, *m_copy = nullptr;
                float* fw = a.W_final[i] ? a.W_final[i] + (size_t)seq * dh : nullptr;
                float* fm = a.W_final[i] ? a.M_final[i] + (size_t)seq * dh : nullptr;
                if (a.save_states == 1) {
                    float* ck = ws + lay.ckpt + (size_t)(c + 1) * 2 * NMAT * dh;
                    w_out = ck + (size_t)i * dh; m_out = ck + (size_t)(NMAT + i) * dh;
                    if (last_chunk && fw) { w_copy = fw; m_copy = fm; }
                } else if (last_chunk && fw) {
                    if (normed) { w_copy = fw; m_copy = fm; }
                    else { w_out = fw; m_out = fm; }
                } else if (a.save_states == 2 && (c + 1) % lay.seg == 0) {
                    float* ck = ws + lay.cck + (size_t)((c + 1) / lay.seg) * 2 * NMAT * dh;
                    w_copy = ck + (size_t)i * dh; m_copy = ck + (size_t)(NMAT + i) * dh;
                }
                // lanes and columns are (d, hidden units) for the first matrices, (hidden units, d) for the last
                const int ln_lim = i < LAST ? d : min(two ? 128 : 64, h - b0 * 64), es = i < LAST ? d : h;
                bool waited = false;
#pragma unroll 1
                for (int half = 0; half < 2; ++half) {
                    const int col = 32 * grp + 16 * half;
                    if (i < LAST ? col >= 64 && !two : col >= dp) break;
                    const int nj = i < LAST ? h - b0 * 64 - col : d - col;
                    const size_t base = i < LAST ? (size_t)(b0 * 64 + col) * d : (size_t)col * h + b0 * 64;
                    float w[16], m[16], acc[16];
                    const bool lane_ok = row < ln_lim;
                    // indices are clamped and values masked: with a branch at every load they were one round trip each
                    if (nj > 0) {
                        const size_t e = base + min(row, ln_lim - 1);
#pragma unroll
                        for (int j = 0; j < 16; ++j) w[j] = w_in[e + (size_t)(min(j, nj - 1) * es)];
                        if (m_in)
#pragma unroll
                            for (int j = 0; j < 16; ++j) m[j] = m_in[e + (size_t)(min(j, nj - 1) * es)];
                        else
#pragma unroll
                            for (int j = 0; j < 16; ++j) m[j] = 0.0f;
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; ++j) w[j] = m[j] = 0.0f;
                    }
                    if (!waited) await(&sh.acc_full, bit(kAcc), 531);
                    waited = true;
                    acc16(lanes + 128 + col, acc);  // G_t = -grad: the aggregations enter with a minus sign
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float mj = m[j];
                        m[j] = cb * mj - acc[j];
                        w[j] = cw * w[j] + cm * mj;
                    }
                    acc16(lanes + col, acc);
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const bool ok = lane_ok && j < nj;
                        w[j] = ok ? w[j] - acc[j] : 0.0f;
                        const size_t e = base + row + (size_t)(j * es);
                        if (ok) {
                            w_out[e] = w[j]; m_out[e] = m[j];
                            if (w_copy) { w_copy[e] = w[j]; m_copy[e] = m[j]; }
                        }
                    }
                    if (!normed && (i < LAST ? row < dp : row < 64 || two)) {
                        const int hblk = b0 + ((i < LAST ? col : row) >> 6), dblk = (i < LAST ? row : col) >> 6;
                        st_split16(blk(wb_of(i, c + 1)) + ((size_t)hblk * db + dblk) * B, row & 63, col & 63, w);
                    }
                }
                if (!waited) await(&sh.acc_full, bit(kAcc), 532);
                par ^= kAcc;
                arrive1(&sh.tile_free);
                release(&sh.acc_free);
            } else {
                // ---- every row w of every W_i becomes n w / (||w|| + eps_n), one warp per row; then the operand blocks of the result
                const int i = it.part < LAST * ns ? it.part / ns : LAST, part = it.part - i * ns;
                const int r0 = i < LAST ? part * 128 : part * 64, rows = i == LAST ? d : h, cols = i == LAST ? h : d;
                const int r1 = min(rows, r0 + (i < LAST ? 128 : 64)), maxdim = d > h ? d : h;
                await(&sh.go[n & 1], n >> 1, 533);
                float* w0 = a.save_states == 1 ? ws + lay.ckpt + (size_t)(c + 1) * 2 * NMAT * dh + (size_t)i * dh : ws + lay.W[i];
                float* w_copy = last_chunk && a.W_final[i] ? a.W_final[i] + (size_t)seq * dh : nullptr;
                const float* target = a.row_norm[i] + (size_t)seq * rows;
                for (int r = r0 + warp; r < r1; r += kEpiWarps) {
                    float* w = w0 + (size_t)r * cols;
                    float ss = 0.0f;
                    for (int j = lane; j < cols; j += 32) ss += w[j] * w[j];
                    const float nrm = sqrtf(warp_sum(ss)), g = target[r] / (nrm + a.norm_eps);
                    for (int j = lane; j < cols; j += 32) {
                        w[j] *= g;
                        if (w_copy) w_copy[(size_t)r * cols + j] = w[j];
                    }
                    if (a.save_states && lane == 0) ws[lay.rown + ((size_t)c * 3 + i) * maxdim + r] = nrm;
                }
                epi_sync();
                if (!last_chunk) {
                    if (i < LAST) matrix_to_blocks(w0, d, h, 0, db, 2 * part, min(hb, 2 * part + 2), blk(wb_of(i, c + 1)), 1, db, warp, kEpiWarps, lane);
                    else matrix_to_blocks(w0, h, d, 0, hb, part, part + 1, blk(wb_of(i, c + 1)), db, 1, warp, kEpiWarps, lane);
                }
                arrive1(&sh.tile_free);
                arrive1(&sh.side_free);
                await(&sh.side_free, n, 534);  // the MMA warp, which has nothing to do here, has seen the item too
                release(&sh.acc_free);
            }
            fence_proxy_async_all();
            arrive1(&sh.written[n & 1]);
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (sh.dead) {  // a wait has given up: copies nobody waited for may still be under way
        const long long t0 = clock64();
        while (clock64() - t0 < 8000000) {}
        __syncthreads();
    }
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// Operand blocks of the first chunk's weights, its scalar kernels, the initial state into the saved slots; counters to 0
template <int NMAT> __global__ void __launch_bounds__(256) tile_flow_init_kernel(const SimtFwdArgs a) {
    const SimtLayout& lay = a.lay;
    const TileLayout& tl = lay.tl;
    const int seq = blockIdx.x, d = a.d, h = a.h, lane = threadIdx.x & 31, w = blockIdx.y * 8 + (threadIdx.x >> 5), nw = gridDim.y * 8;
    const size_t dh = (size_t)d * h;
    float* ws = reinterpret_cast<float*>(a.ws) + (size_t)seq * lay.per_seq;
    const float* ck0 = a.init_slot >= 0 ? ws + lay.cck + (size_t)a.init_slot * 2 * NMAT * dh : nullptr;
    float* ck = a.save_states ? ws + (a.save_states == 1 ? lay.ckpt : lay.cck) : nullptr;
    if (blockIdx.y == 0) {
        if (threadIdx.x == 0) *reinterpret_cast<Counters*>(ws + tl.fred) = Counters{};
        const size_t t = (size_t)seq * a.Ls;
        if (threadIdx.x < 32) chunk_scalars_warp<float>(a.eta + t, a.beta + t, a.gamma + t, min(a.C, a.L), reinterpret_cast<ChunkScalars<float>*>(ws + tl.fslot));
    }
#pragma unroll
    for (int i = 0; i < NMAT; ++i) {
        const float* wi = ck0 ? ck0 + (size_t)i * dh : a.W_init[i] + (size_t)seq * dh;
        const float* mi = ck0 ? ck0 + (size_t)(NMAT + i) * dh : (a.M_init[i] ? a.M_init[i] + (size_t)seq * dh : nullptr);
        unsigned char* to = reinterpret_cast<unsigned char*>(ws + tl.Wb[i]);
        if (i < NMAT - 1) matrix_to_blocks(wi, d, h, 0, tl.db, 0, tl.hb, to, 1, tl.db, w, nw, lane);
        else matrix_to_blocks(wi, h, d, 0, tl.hb, 0, tl.db, to, tl.db, 1, w, nw, lane);
        if (ck && ck != ck0)
            for (size_t e = (size_t)blockIdx.y * 256 + threadIdx.x; e < dh; e += (size_t)gridDim.y * 256) {
                ck[i * dh + e] = wi[e];
                ck[(NMAT + i) * dh + e] = mi ? mi[e] : 0.0f;
            }
    }
}

template <int KIND, bool WIDE> int launch(const SimtFwdArgs& a, cudaStream_t st) {
    constexpr int NMAT = KIND == 0 ? 2 : 3;
    static bool attr_done[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return (int)cudaGetLastError();
    if (dev < 0 || dev >= 64 || !attr_done[dev]) {
        cudaError_t e = cudaFuncSetAttribute(tile_flow_kernel<KIND, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFlowSmem);
        if (e != cudaSuccess) return (int)e;
        if (dev >= 0 && dev < 64) attr_done[dev] = true;
    }
    const FlowArgs f{a, flow_plan(a.lay.tl, a.N, a.L, a.C, NMAT, a.row_norm[0] != nullptr)};
    const int per = (296 + a.N - 1) / a.N;
    tile_flow_init_kernel<NMAT><<<dim3(a.N, per < 16 ? per : 16), 256, 0, st>>>(a);
    const long long items = (long long)a.N * f.p.slots;
    tile_flow_kernel<KIND, WIDE><<<items < 148 ? (int)items : 148, kFlowThreads, kFlowSmem, st>>>(f);
    return (int)cudaGetLastError();
}

}  // namespace

int tile_flow_launch(const SimtFwdArgs& a, int kind, void* stream) {
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (a.lay.tl.hb > 2 * kUSteps) return kind == 0 ? launch<0, true>(a, st) : launch<1, true>(a, st);
    return kind == 0 ? launch<0, false>(a, st) : launch<1, false>(a, st);
}

}  // namespace e2ttt
