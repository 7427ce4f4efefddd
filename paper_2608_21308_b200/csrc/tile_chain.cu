// The serial part of the block-tiled reverse pass (tile_bwd.cu) with the adjoint T of the weights on chip.
//
// What bounds the chain: the adjoints T, S of the state are read and written in every chunk, as fp32 masters and as operand blocks;
// through the workspace that was 7 of 10.7 MB of memory traffic per chunk and sequence at d = 128, h = 512, C = 64, and with 64
// sequences at once it does not fit L2.  Here a cluster has one CTA per 128 hidden units (33 clusters of 4 fit the GPU; one CTA per
// 64 units was slower: 15 clusters of 8), and a CTA keeps its slices for the whole launch:
//   tensor memory : fp32 masters of T, 128 x 128 per matrix.  The contiguous index of the matrix in memory is on the lanes (d for the
//                   first matrices, hidden units for the last), so that the state (T, S, and the saved W, M of every chunk) is read
//                   and written whole lines at a time
//   shared memory : operand blocks (hi, lo) of T of as many matrices as fit 128 KB (two at d > 64), rows = the index on the
//                   lanes: read K-major with that index on the lanes, MN-major with the other one there
// S, and T blocks that do not fit, live in the workspace; 33 sequences' worth stays in L2.
// A chunk starts with one pass over the masters (T <- cw T, S <- cm T + cb S; the blocks of the new S go to the other of two buffers,
// by the parity of the chunk) while the first products run on the operand blocks of the arriving T, S.  Every product that contributes
// to T has an epilogue of its own, which adds it to the master; after a matrix's last one T's operand blocks are written anew.
// Everything else streams from the slots that tile_prep and tile_rec filled.
//
// 18 warps: 0-15 epilogues (warp w: lanes 32 (w & 3).., group w >> 2 of the columns), 16 copies operand blocks, 17 issues MMAs; with the GELU
// network two more, for the barriers alone (chain_threads).
#include <type_traits>

#include "tile_rec.cuh"

namespace e2ttt {
using namespace tile;

namespace {

// GELU network: two more warps make up the copy and MMA warps' warpgroup, so that setmaxnreg can give the epilogues their registers (104,
// and nothing spills: 64 sequences of 64 chunks 9.07 -> 8.40 ms).  The SwiGLU epilogues spill either way, and the copy and MMA warps of
// that network as well with 64 (one chunk of 512 tokens, 32 sequences 559 -> 582 us)
constexpr int chain_threads(int kind) { return kind == 0 ? 640 : kThreads; }
constexpr int kCells = 6;                        // operand ring, cells of 16 KB; a load takes one or two neighbouring ones
constexpr uint32_t kCell = 2 * kHalf;
constexpr int kLoads = 8;                        // loads in flight at most
// Shared memory: resident operands | ring | ChainShared.  An MMA covers 128 lanes: of a single-block lane-side operand it reads 8 KB
// more than there is (lanes whose results nobody reads), so such a load takes two cells.
constexpr uint32_t kResident = 128 * 1024, kRingBytes = kCells * kCell;

struct ChainShared {
    uint64_t full[kLoads], empty[kLoads], acc_full[2], acc_empty[2];
    // once per chunk: operand blocks of T, S written; phb written; masters scaled; zb written
    uint64_t ops, phb, scaled, zb;
    uint32_t tmem;
    int dead;
    float dots[2][16][4];  // by the parity of the launch's chunk: a warp may be a chunk's scaling ahead of the one that adds them up
    float kb[16][32];  // per epilogue warp: K^W then K^M of its 16 tokens of the current block of 64; normalisation: scratch
};
constexpr size_t kChainSmem = kResident + kRingBytes + sizeof(ChainShared);
static_assert(kChainSmem <= 232448 && kRecSmem <= kChainSmem, "227 KB of shared memory per CTA");

__device__ __forceinline__ uint32_t cells_of(const Opnd& o, bool lane_side) { return (o.lo && o.p1) || (lane_side && !o.p1) ? 2u : 1u; }
__device__ __forceinline__ uint32_t lo_of(const Opnd& o) { return o.p1 ? kCell : kHalf; }  // hi blocks first, then lo blocks

// An operand in shared memory as the MMAs see it
struct SOp {
    uint32_t addr, lo;  // hi part; distance to the lo part, 0: none
    uint32_t lbo;       // MN-major: distance between the slabs of 64 M / N indices
    bool mn, wide;      // MN-major; 128 (else 64) columns when it is the column side
};

template <int NSET> struct Chain {
    uint32_t resident, ring;
    ChainShared* sh;
    uint32_t tmem;
    WaitCtx wc;
    int warp, lane, nranks;
    uint32_t load_no = 0, cell = 0;           // ring: next load, next free cell
    uint32_t flying = 0, used = 0, feet = 0;  // copy warp: loads not known to be consumed, their cells, footprints (2 bits each)
    uint32_t job = 0;
    bool own_T = false;

    __device__ bool epi() const { return warp < 16; }
    __device__ bool copier() const { return warp == 16; }
    __device__ bool issuer() const { return warp == 17; }

    __device__ void setup(unsigned char* smem, ChainShared* s, int* status, int nranks_) {
        resident = smem_u32(smem);
        ring = resident + kResident;
        sh = s;
        warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);  // (as in Engine: uniform for the compiler)
        lane = threadIdx.x & 31;
        nranks = nranks_;
        if (threadIdx.x == 0) {
            for (int i = 0; i < kLoads; ++i) { mbar_init(&s->full[i], 1); mbar_init(&s->empty[i], 1); }
            for (int i = 0; i < 2; ++i) { mbar_init(&s->acc_full[i], 1); mbar_init(&s->acc_empty[i], 16); }
            mbar_init(&s->ops, 16); mbar_init(&s->phb, 16); mbar_init(&s->scaled, 16); mbar_init(&s->zb, 16);
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
    // What threads write (shared memory or workspace) is read by MMAs and bulk copies, through the async proxy
    __device__ void cluster_arrive_all() {
        fence_proxy_async_all();
        tc_fence_before_sync();
        __syncwarp();
        if (nranks > 1) cluster_arrive();
    }
    __device__ void cluster_wait_all() {
        if (nranks > 1) cluster_wait();
        else __syncthreads();
        tc_fence_after_sync();
        fence_proxy_async_all();
    }
    // Epilogue warps: this warp's part of what `bar` stands for is written.  A fence of global memory waits for all stores under way
    // (2-3 thousand cycles of a chunk each).  The blocks of the new S, behind `scaled`, are loaded after the chunk's cluster barriers, whose
    // fence is in time for them; `ops` needs none where all of T's blocks are in shared memory (`own_T`)
    __device__ void signal(uint64_t* bar) {
        if (bar == &sh->ops && own_T) fence_proxy_async_smem();
        else if (bar != &sh->scaled) fence_proxy_async_all();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar);
    }
    __device__ void await(uint64_t* bar, uint32_t phase, int where) {
        mbar_wait(bar, phase & 1, wc, where);
        tc_fence_after_sync();
        fence_proxy_async_all();
    }
    static __device__ void epi_sync() { asm volatile("bar.sync 1, 512;" ::: "memory"); }

    __device__ uint32_t place(uint32_t n) {  // two cells do not wrap around
        if (n == 2 && cell % kCells == kCells - 1) ++cell;
        const uint32_t at = cell;
        cell += n;
        return (at % kCells) * kCell;
    }
    __device__ void load(const Opnd& o, int k, bool lane_side) {  // copy warp
        const uint32_t before = cell, at = place(cells_of(o, lane_side)), foot = cell - before;
        while (flying > 0 && (used + foot > kCells || flying == kLoads)) {
            const uint32_t oldest = load_no - flying;
            mbar_wait(&sh->empty[oldest % kLoads], (oldest / kLoads) & 1, wc, 401);
            used -= feet & 3;
            feet >>= 2;
            --flying;
        }
        feet |= foot << (2 * flying++);
        used += foot;
        uint64_t* full = &sh->full[load_no % kLoads];
        ++load_no;
        if (lane == 0) {
            const uint32_t dst = ring + at;
            const size_t off = (size_t)k * o.ks;
            mbar_expect_tx(full, kHalf * (o.p1 ? 2u : 1u) * (o.lo ? 2u : 1u));
#pragma unroll 1
            for (int part = 0; part < (o.lo ? 2 : 1); ++part) {
                bulk_g2s(dst + part * lo_of(o), o.p0 + off + part * kHalf, kHalf, full);
                if (o.p1) bulk_g2s(dst + part * lo_of(o) + kHalf, o.p1 + off + part * kHalf, kHalf, full);
            }
        }
        __syncwarp();
    }
    __device__ SOp take(const Opnd& o, uint32_t& bar, bool lane_side) {  // MMA warp: the next load, once it is there
        const uint32_t at = place(cells_of(o, lane_side));
        bar = load_no % kLoads;
        mbar_wait(&sh->full[bar], (load_no / kLoads) & 1, wc, 402);
        ++load_no;
        tc_fence_after_sync();
        return {ring + at, o.lo ? lo_of(o) : 0u, kHalf, o.mn, o.p1 != nullptr};
    }
    // D (+)= A B^T over 64 k
    __device__ void mma(uint32_t d, const SOp& a, const SOp& b, bool acc) {
        const uint32_t idesc = make_idesc(128, b.wide ? 128 : 64, a.mn, b.mn);
        const uint32_t sa = a.mn ? 2048u : 32u, sb = b.mn ? 2048u : 32u;
#pragma unroll 1
        for (int ks = 0; ks < 4; ++ks) {
            const uint64_t ah = make_smem_desc(a.addr + ks * sa, a.lbo, 1024), bh = make_smem_desc(b.addr + ks * sb, b.lbo, 1024);
            bool c = acc || ks > 0;
            if (a.lo) { umma_bf16_elect(d, ah + (a.lo >> 4), bh, idesc, c, lane == 0); c = true; }  // small terms first
            if (b.lo) { umma_bf16_elect(d, ah, bh + (b.lo >> 4), idesc, c, lane == 0); c = true; }
            umma_bf16_elect(d, ah, bh, idesc, c, lane == 0);
        }
    }
    __device__ uint32_t acc() const { return NSET == 2 ? 256 + (job & 1) * 128 : 384; }  // first column of the job's accumulators
    __device__ void job_begin() {
        if (issuer()) {
            if (job >= NSET) mbar_wait(&sh->acc_empty[job % NSET], ((job / NSET) - 1) & 1, wc, 403);
            tc_fence_after_sync();
        }
    }
    __device__ void job_end() {  // copy and MMA warps
        if (issuer()) umma_commit_elect(&sh->acc_full[job % NSET], lane == 0);
        ++job;
    }
    // One product over nk slices of 64, copy and MMA warps.  Paired: the column-side operand x with two lane-side partners,
    // D[col] += Y X^T and D[col + 64] += Z X^T, where Y is resident or from the ring; else D[col] += X Z^T with x on the lane side.
    // All products of a chunk go through the one copy of this code: with a copy for each, the two warps pushed the epilogues out of
    // the instruction cache in every chunk (a quarter of all warps' time).
    struct Product {
        int nk;
        Opnd x, y, z;
        SOp part;             // Y, where it is resident (x ring otherwise), and its step per slice
        uint32_t part_step, col;
        bool paired, resident, acc0;
        uint64_t* before;     // what the copy warp waits for between the first load of x and the first of z
        bool before_cluster;  // the cluster barrier instead
    };
    __device__ void run(const Product& P, uint32_t phase) {
        if (copier()) {
#pragma unroll 1
            for (int k = 0; k < P.nk; ++k) {
                load(P.x, k, !P.paired);
                if (k == 0 && P.before) await(P.before, phase, 406);
                if (k == 0 && P.before_cluster) cluster_wait_all();
                if (P.paired && !P.resident) load(P.y, k, true);
                load(P.z, k, P.paired);
            }
        } else if (issuer()) {
#pragma unroll 1
            for (int k = 0; k < P.nk; ++k) {
                uint32_t bx, by, bz;
                const bool c = P.acc0 || k > 0;
                const SOp x = take(P.x, bx, !P.paired);
                if (P.paired) {
                    SOp y = P.part;
                    y.addr += k * P.part_step;
                    if (!P.resident) y = take(P.y, by, true);
                    mma(P.col, y, x, c);
                    if (!P.resident) umma_commit_elect(&sh->empty[by], lane == 0);
                }
                const SOp z = take(P.z, bz, P.paired);
                mma(P.col + (P.paired ? 64 : 0), P.paired ? z : x, P.paired ? x : z, c);
                umma_commit_elect(&sh->empty[bx], lane == 0);
                umma_commit_elect(&sh->empty[bz], lane == 0);
            }
        }
    }
    template <typename F> __device__ void job_out(F f) {  // epilogue warps
        mbar_wait(&sh->acc_full[job % NSET], (job / NSET) & 1, wc, 404);
        tc_fence_after_sync();
        f(tmem + acc() + ((uint32_t)(32 * (warp & 3)) << 16));
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh->acc_empty[job % NSET]);
        ++job;
    }
};

__device__ __forceinline__ void acc_st16(uint32_t t, const float (&v)[16]) {
    uint32_t r[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) r[j] = __float_as_uint(v[j]);
    tmem_st16(t, r);
}

// BESIDE: the launch has CTAs for the next group; without them the chain keeps the registers that its code costs (2 % of the time).
// One sequence of 8192 tokens x 16 heads, training step: 12.8 -> 11.9 ms
template <int KIND, bool NORMED, bool BESIDE> __global__ void __launch_bounds__(chain_threads(KIND), 1)
tile_chain_kernel(const GroupArgs ga, const NextGroup next) {
    constexpr int NMAT = (KIND == 0) ? 2 : 3, LAST = NMAT - 1;
    constexpr bool SW = KIND == 1;
    extern __shared__ __align__(1024) unsigned char chain_smem[];
    ChainShared& sh = *reinterpret_cast<ChainShared*>(chain_smem + kResident + kRingBytes);
    const SimtBwdArgs& a = ga.a;
    if (BESIDE && (int)blockIdx.x >= a.N * a.cl) {  // SMs without a part in the chain: what the next group does not need T, S for
        rec_items<KIND>(a, next, chain_smem, blockIdx.x - a.N * a.cl, gridDim.x - a.N * a.cl);
        return;
    }
    const int CL = a.cl, seq = blockIdx.x / CL, rank = blockIdx.x % CL;
    constexpr int EARLY = SW ? 1 : 2;  // accumulator sets
    Chain<EARLY> G;
    G.setup(chain_smem, &sh, a.status, CL);
    const int warp = G.warp, lane = G.lane;
    const SimtLayout& lay = a.lay;
    const TileLayout& tl = lay.tl;
    const int d = a.d, h = a.h, db = tl.db, tb = tl.tb, dp = db * 64;
    const size_t dh = (size_t)d * h;
    const int b0 = 2 * rank, h0 = b0 * 64, nh = min(128, h - h0);  // own hidden blocks and units
    const bool two = b0 + 1 < tl.hb;
    const int nb = two ? 2 : 1;
    float* ws = reinterpret_cast<float*>(a.ws) + (size_t)seq * lay.per_seq;
    auto blk = [&](size_t off) { return bytes_of(ws + off); };
    const size_t sblks = (size_t)db * tl.hb * kTileBlk;  // between the two buffers of S blocks
    // resident T of matrix i at i * unit: hi blocks, then lo; blocks that share the index on their columns are neighbours
    const uint32_t half = 2u * db * kHalf, unit = 2 * half;
    const int nres = min(NMAT, (int)(kResident / unit));

    if (!G.epi()) {
        // ================================================================= copy and MMA warps
        if (!SW) asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        if (warp > 17) {  // the barriers of all threads
#pragma unroll 1
            for (int g = 0; g < ga.ng * (NORMED ? 3 : 2) + 1; ++g) {
                G.cluster_arrive_all();
                G.cluster_wait_all();
            }
            G.teardown();
            return;
        }
        // blocks of a [hidden x d] family in the workspace, own hidden units: hidden units on the lanes (MN-major where the rows are d),
        // contraction over d; and d on the lanes, contraction over the hidden units
        auto w_by_h = [&](const unsigned char* m, bool rows_d) {
            const unsigned char* p = m + (size_t)b0 * db * B;
            return Opnd{p, two ? p + (size_t)db * B : nullptr, B, true, rows_d};
        };
        auto w_by_d = [&](const unsigned char* m, bool rows_d) {
            const unsigned char* p = m + (size_t)b0 * db * B;
            return Opnd{p, db == 2 ? p + B : nullptr, (uint32_t)db * B, true, !rows_d};
        };
        size_t sbuf = 0;  // S blocks of the chunk at hand
        using Product = typename Chain<EARLY>::Product;
        // products of a [tokens x ..] operand with T and S of matrix i, hidden units or d on the lanes
        auto by_h = [&](Product& P, const Opnd& x, int i) {
            const bool f = i < LAST;
            P.nk = db;
            P.x = x;
            P.paired = true;
            P.resident = i < nres;
            P.part = SOp{G.resident + i * unit, half, f ? db * kHalf : kHalf, f, false};
            P.part_step = f ? kHalf : 2 * kHalf;
            P.y = w_by_h(blk(tl.Tb[i]), f);
            P.z = w_by_h(blk(tl.Sb[i] + sbuf), f);
        };
        auto by_d = [&](Product& P, const Opnd& x, int i) {
            const bool f = i < LAST;
            P.nk = nb;
            P.x = x;
            P.paired = true;
            P.resident = i < nres;
            P.part = SOp{G.resident + i * unit, half, f ? kHalf : 2 * kHalf, !f, false};
            P.part_step = f ? db * kHalf : kHalf;
            P.y = w_by_d(blk(tl.Tb[i]), f);
            P.z = w_by_d(blk(tl.Sb[i] + sbuf), f);
        };
        auto simple = [](Product& P, int nk, const Opnd& x, const Opnd& z) {
            P.nk = nk;
            P.x = x;
            P.z = z;
        };
        // What a chunk reads was written long ago and comes from HBM: into L2 half a chunk ahead (a whole chunk ahead would not fit
        // beside the state of 33 sequences)
        auto pf = [&](const void* p, size_t bytes) {
            if (((reinterpret_cast<size_t>(p) | bytes) & 15) == 0) l2_prefetch(p, (uint32_t)bytes);
        };
        const size_t own = (size_t)b0 * tb * 4096, own_bytes = (size_t)nb * tb * B;
        auto prefetch_early = [&](int g) {  // for the products with T, S and their epilogues
            float* sn = slot_of(a, seq, ga.s0 + g);
            if (lane < 6) {
                const size_t src[6] = {tl.sph, tl.sc1, tl.sc4, tl.sAk, tl.sPz[0], SW ? tl.sPz[LAST - 1] : tl.sAk};
                pf(sn + src[lane] + own, own_bytes);
            } else if (lane < 8 && SW) {
                pf(sn + (lane == 6 ? tl.sc2 : tl.sg1) + own, own_bytes);
            } else if (lane >= 8 && lane < 11) {
                const size_t src[3] = {tl.sK, tl.sPu, tl.spu};
                if ((lane - 8) % CL == rank) pf(sn + src[lane - 8], (size_t)tb * 64 * dp * (lane == 8 ? 2 : 4));
            } else if (lane == 11) {
                pf(sn + tl.sW[LAST] + (size_t)b0 * db * kTileBlk, (size_t)nb * db * B);
            }
            __syncwarp();
        };
        auto prefetch_late = [&](int g) {  // for the rest of the chunk
            float* sn = slot_of(a, seq, ga.s0 + g);
            if (lane < 3) {
                const size_t src[3] = {tl.sAq, tl.sZq[0], SW ? tl.sZq[LAST - 1] : tl.sAq};
                pf(sn + src[lane] + own, own_bytes);
            } else if (lane >= 4 && lane < 4 + LAST) {
                pf(sn + tl.sW[lane - 4] + (size_t)b0 * db * kTileBlk, (size_t)nb * db * B);
            } else if (lane >= 8 && lane < 11) {
                const size_t src[3] = {tl.sQ, tl.sUq, tl.sy};
                if ((lane - 8) % CL == rank) pf(sn + src[lane - 8], (size_t)tb * 64 * dp * (lane == 8 ? 2 : 4));
            }
            __syncwarp();
        };
        // The saved W, M that the scaling of the masters reads: plain prefetches, which do not stand in the bulk engine's queue before
        // the loads of the products
        auto prefetch_state = [&](int g) {
            const float* cn = ws + lay.ckpt + (size_t)(ga.c0 + g) * 2 * NMAT * dh;
            auto line = [](const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); };
            for (int i = 0; i < 2 * LAST; ++i) {
                const float* p = cn + (size_t)((i & 1 ? NMAT : 0) + (i >> 1)) * dh + (size_t)h0 * d;
                for (int r = 32 * lane; r < nh * d; r += 32 * 32) line(p + r);
            }
            const float* wl = cn + (size_t)LAST * dh + h0;
            for (int r = lane; r < 8 * d; r += 32)
                if ((r & 3) * 32 < nh) line(wl + (size_t)(r & 4 ? NMAT : 0) * dh + (size_t)(r >> 3) * h + (r & 3) * 32);
            __syncwarp();
        };
        uint32_t n = 0;
        if (G.copier()) prefetch_state(ga.ng - 1);
        for (int g = ga.ng - 1; g >= 0; --g, ++n) {
            const int c = ga.c0 + g, len = min(a.C, a.L - c * a.C), tbn = (len + 63) / 64;
            float* sl = slot_of(a, seq, ga.s0 + g);
            auto sblk = [&](size_t off) { return bytes_of(sl + off); };
            auto tok_h = [&](const unsigned char* m, int tk) { return Opnd{m + ((size_t)b0 * tb + tk) * B, nullptr, (uint32_t)tb * B, true, true}; };
            auto h_tok = [&](const unsigned char* m) {
                const unsigned char* p = m + (size_t)b0 * tb * B;
                return Opnd{p, two ? p + (size_t)tb * B : nullptr, B, true, false};
            };
            auto tok_d = [&](const unsigned char* m) { return Opnd{m, db == 2 ? m + B : nullptr, (uint32_t)db * B, true, true}; };
            auto key_d = [&](const unsigned char* m) { return Opnd{m, db == 2 ? m + kHalf : nullptr, (uint32_t)db * kHalf, false, true}; };

            sbuf = (c & 1) * sblks;
            if (NORMED) {
                G.cluster_arrive_all();
                G.cluster_wait_all();
            }
            G.cluster_arrive_all();  // the first of the chunk's two barriers: nothing of these warps' is waited for
            // T in shared memory waits for the blocks written at the end of the chunk before; loads of S only for its scaling there,
            // which the copy warp waits for inside that chunk
            if (G.issuer() || n == 0) G.await(&sh.ops, n, 405);
            // Steps of the chunk: phase, block of 64 tokens, product
            //   0  everything with T, S          3  adjoint of u back through W_last
            //   1  pub += W_last phb             5  dk += W_first^T zb
            //   2, 4, 6  contributions to T: q zq (first matrices), aq uq, phb pu and ak uk (last), zb k (first).  The first ones wait for
            //      no rows: as many as there are accumulator sets run while the rows do
#pragma unroll 1
            for (int ph = 0; ph < 7; ++ph) {
                if (ph == 1 && G.copier()) {
                    prefetch_late(g);
                    if (g > 0) prefetch_state(g - 1);
                }
                if (ph == 3) {
                    // Taken before the loads that the chunk's end waits for: later, the epilogues could be through with the next chunk's
                    // scaling, and a wait for this one's parity would be a wait for the one after
                    if (G.copier()) G.await(&sh.scaled, n, 410);
                    G.cluster_wait_all();
                    G.cluster_arrive_all();
                    if (G.issuer()) G.cluster_wait_all();
                }
                const int ntk = ph == 2 || ph == 4 || ph == 6 ? 1 : tbn;
                const int nstep = ph == 0 ? 2 * LAST + 2 : ph == 2 ? EARLY : ph == 4 ? LAST + 3 - EARLY : ph >= 5 ? LAST : 1;
#pragma unroll 1
                for (int e = 0, tk = 0, st = 0; e < ntk * nstep; ++e) {
                    if (ph == 0 && st == LAST && tk == 0 && nres < NMAT && G.copier()) G.await(&sh.ops, n, 411);
                    // the first matrices' dk products of phases 0 and 5 share a job
                    const bool opens = ph == 0 ? st <= LAST + 2 : ph == 5 ? st == 0 : true, closes = ph == 0 ? st < LAST + 2 || st == 2 * LAST + 1 : ph == 5 ? st == nstep - 1 : true;
                    Product P{};
                    P.col = G.tmem + G.acc();
                    P.acc0 = !opens;
                    if (ph == 0) {
                        if (st < LAST) by_h(P, Opnd{sblk(tl.sK) + (size_t)tk * db * kHalf, nullptr, kHalf, false, false}, st);
                        else if (st == LAST) by_h(P, Opnd{sblk(tl.sPu) + (size_t)tk * db * B, nullptr, B, true, false}, LAST);
                        else if (st == LAST + 1) by_d(P, tok_h(sblk(tl.sAk), tk), LAST);
                        else by_d(P, tok_h(sblk(tl.sPz[st - LAST - 2]), tk), st - LAST - 2);
                    } else if (ph == 1) {
                        simple(P, nb, w_by_d(sblk(tl.sW[LAST]), false), tok_h(blk(tl.bPhb), tk));
                        P.before = &sh.phb;
                    } else if (ph == 2 || ph == 4) {
                        const int k = ph == 2 ? st : EARLY + st;
                        if (k < LAST) simple(P, tbn, key_d(sblk(tl.sQ)), h_tok(sblk(tl.sZq[k])));
                        else if (k == LAST) simple(P, tbn, h_tok(sblk(tl.sAq)), tok_d(sblk(tl.sUq)));
                        else if (k == LAST + 1) simple(P, tbn, h_tok(blk(tl.bPhb)), tok_d(sblk(tl.sPu)));
                        else simple(P, tbn, h_tok(sblk(tl.sAk)), tok_d(blk(tl.bUk)));
                    } else if (ph == 3) {
                        simple(P, db, w_by_h(sblk(tl.sW[LAST]), false), Opnd{blk(tl.bUk) + (size_t)tk * db * B, nullptr, B, true, false});
                        P.before_cluster = tk == 0;
                    } else if (ph == 5) {
                        simple(P, nb, w_by_d(sblk(tl.sW[st]), true), tok_h(blk(tl.bZk[st]), tk));
                        P.before = &sh.zb;
                    } else {
                        simple(P, tbn, key_d(sblk(tl.sK)), h_tok(blk(tl.bZk[st])));
                    }
                    if (opens) G.job_begin();
                    G.run(P, n);
                    if (closes) G.job_end();
                    if (++st == nstep) { st = 0; ++tk; }
                }
            }
            if (G.copier() && g > 0) prefetch_early(g - 1);
        }
        G.cluster_arrive_all();
        G.cluster_wait_all();
        G.teardown();
        return;
    }

    // ===================================================================== epilogue warps
    if (!SW) asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
    const int q4 = warp & 3, grp = warp >> 2, row = 32 * q4 + lane;
    const bool on_h = row < 64 || two;      // lane of a product with hidden units on the lanes
    const int bl = b0 + (row >> 6);         // its hidden block
    const uint32_t lanes = G.tmem + ((uint32_t)(32 * q4) << 16);
    // A master is handled in pieces of 16 columns: piece pc of this warp = columns 32 grp + 16 pc ..  Lanes and columns are (d, hidden
    // units) for the first matrices, (hidden units, d) for the last
    auto col_of = [&](int pc) { return 32 * grp + 16 * pc; };
    auto lane_lim = [&](int i) { return i < LAST ? d : nh; };
    auto col_lim = [&](int i) { return i < LAST ? nh : d; };
    auto mask = [&](int i, int col, float (&v)[16]) {  // whatever lies outside the real matrix -> 0
        const int nc = col_lim(i) - col;
        if (row >= lane_lim(i) || nc < 16)
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = row < lane_lim(i) && j < nc ? v[j] : 0.0f;
    };
    // operand blocks of T (resident or not) and S (of the chunks of one parity): 16 values of row `row`
    auto put = [&](bool is_T, int sbuf, int i, int col, const float (&v)[16]) {
        const int rb = row >> 6, cb = col >> 6;
        if (i < LAST ? (row >= dp || (cb && !two)) : (!on_h || col >= dp)) return;
        const uint32_t res = i < LAST ? (uint32_t)(cb * db + rb) : (uint32_t)(cb * 2 + rb);
        if (is_T && i < nres) sts_split16(G.resident + i * unit + res * kHalf, half, row & 63, col & 63, v);
        else {
            const int hblk = i < LAST ? cb : rb, dblk = i < LAST ? rb : cb;
            st_split16(blk(is_T ? tl.Tb[i] : tl.Sb[i] + sbuf * sblks) + (size_t)((b0 + hblk) * db + dblk) * B, row & 63, col & 63, v);
        }
    };
    // A piece of a state-shaped fp32 array (row-major [h x d], the last matrix [d x h]); 0 outside.  At the edges indices are clamped
    // and the values masked: with a branch at every load they were one round trip each.  The strides are opaque to the compiler, which
    // otherwise keeps sixteen offsets per stride in registers, and spills: with 227 KB of shared memory in use hardly any L1 is left,
    // so that a spilled value comes from L2
    auto opaque = [](int x) {
        asm volatile("" : "+r"(x));
        return x;
    };
    auto ld_raw = [&](int i, const float* p, int col, float (&v)[16]) {
        const int nc = col_lim(i) - col;
        if (!p || nc <= 0) {
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = 0.0f;
            return;
        }
        const int ld = opaque(i < LAST ? d : h);
        const float* q = p + (i < LAST ? (size_t)(h0 + col) * d : (size_t)col * h + h0) + min(row, lane_lim(i) - 1);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            v[j] = *q;
            if (j + 1 < nc) q += ld;
        }
    };
    auto ld_state = [&](int i, const float* p, int col, float (&v)[16]) {
        ld_raw(i, p, col, v);
        mask(i, col, v);
    };
    auto st_state = [&](int i, float* p, int col, const float (&v)[16]) {
        const int nc = col_lim(i) - col, ld = opaque(i < LAST ? d : h);
        float* q = p + (i < LAST ? (size_t)(h0 + col) * d : (size_t)col * h + h0) + row;
        if (row < lane_lim(i))
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                if (j < nc) *q = v[j];
                q += ld;
            }
    };

    // ---- T -> tensor memory; T, S -> operand blocks; S -> the workspace
    {
        const bool given = ga.first && !a.carry_in;
#pragma unroll 1
        for (int e = 0; e < 2 * NMAT; ++e) {
            const int i = e >> 1, col = col_of(e & 1);
            const float* tf = given ? (a.dW_final[i] ? a.dW_final[i] + (size_t)seq * dh : nullptr) : ws + lay.T[i];
            const float* sf = given ? (a.dM_final[i] ? a.dM_final[i] + (size_t)seq * dh : nullptr) : ws + lay.S[i];
            float t[16], s[16];
            ld_state(i, tf, col, t);
            ld_state(i, sf, col, s);
            acc_st16(lanes + 128 * i + col, t);
            if (!NORMED) put(true, 0, i, col, t);
            if (ga.first) put(false, (ga.c0 + ga.ng - 1) & 1, i, col, s);  // otherwise the launch before this one left them
            if (given) st_state(i, ws + lay.S[i], col, s);
        }
        tmem_wait_st();
        if (!NORMED) G.signal(&sh.ops);
        G.own_T = nres == NMAT;
    }

    // One row of dk of a chunk = its e-adjoint + the CTAs' partial sums, in CTA order
    const int ci = 4 * lane;
    auto dk_row = [&](int s, int t, int buf) {
        if (ci >= dp) return;
        const float4 x = *reinterpret_cast<const float4*>(ws + tl.bEb[buf] + (size_t)t * dp + ci);
        float o[4] = {x.x, x.y, x.z, x.w};
        add_parts<8>(ws + tl.bdk[buf] + (size_t)t * dp + ci, 2 * CL, (size_t)tb * 64 * dp, o);
        st_tok4(reinterpret_cast<__nv_bfloat16*>(a.dk) + ((size_t)seq * a.Ls + s + t) * d, ci, d, o);
    };

    uint32_t n = 0;
    for (int g = ga.ng - 1; g >= 0; --g, ++n) {
        const int c = ga.c0 + g, s = c * a.C, len = min(a.C, a.L - s), tbn = (len + 63) / 64, buf = c & 1;
        float* sl = slot_of(a, seq, ga.s0 + g);
        const ChunkScalars<float>& sc = *reinterpret_cast<const ChunkScalars<float>*>(sl + tl.ssc);
        const float* ck = ws + lay.ckpt + (size_t)c * 2 * NMAT * dh;
        auto partial = [&](size_t base, int part, int tk) { return ws + base + ((size_t)(rank * 2 + part) * tb * 64 + tk * 64 + 16 * grp) * dp + row; };

        if constexpr (NORMED) {
            // T arrives as the adjoint of the normalised chunk-end weights y = n w / (||w|| + eps_n); with y itself (the next
            // chunk's saved start state) and the saved norm:  w_bar = n/(s + eps_n) y_bar - y <y_bar, y> / (n s),  n_bar = <y_bar, y> / n
            const int maxdim = d > h ? d : h;
            const float* nxt = ck + (size_t)2 * NMAT * dh;
            float* scratch = &sh.kb[0][0];  // 512 floats
            auto factors = [&](int i, int r, bool in, float ty, bool report, float& f, float& gy) {
                const int rows = (i == LAST) ? d : h;
                const float nn = in ? a.row_norm[i][(size_t)seq * rows + r] : 0.0f, nrm = in ? ws[lay.rown + ((size_t)c * 3 + i) * maxdim + r] : 0.0f;
                f = in ? nn / (nrm + a.norm_eps) : 0.0f;
                gy = (nn != 0.0f && nrm > 0.0f) ? ty / (nn * nrm) : 0.0f;
                if (report && in && a.d_row_norm[i]) {
                    float* tbar = a.d_row_norm[i] + (size_t)seq * rows + r;
                    const float nb_ = nn != 0.0f ? ty / nn : 0.0f;
                    *tbar = (c == a.nchunks - 1) ? nb_ : *tbar + nb_;
                }
            };
            float t[16], y[16];
            // a row of the first matrices is a hidden unit, of the last an output: a column of the master either way
#pragma unroll 1
            for (int i = 0; i < NMAT; ++i) {
#pragma unroll 1
                for (int pc = 0; pc < 2; ++pc) {
                    ld_state(i, nxt + (size_t)i * dh, col_of(pc), y);
                    acc16(lanes + 128 * i + col_of(pc), t);
                    mask(i, col_of(pc), t);
#pragma unroll
                    for (int j = 0; j < 16; ++j) t[j] *= y[j];
                    const float x = reduce16(t, lane);
                    if ((lane & 1) == 0) scratch[q4 * 128 + col_of(pc) + (lane >> 1)] = x;
                }
                G.epi_sync();
                if (i == LAST) {  // its rows span the cluster
                    if (threadIdx.x < 128)
                        ws[tl.bred + (size_t)rank * 128 + threadIdx.x] = (scratch[threadIdx.x] + scratch[128 + threadIdx.x]) + (scratch[256 + threadIdx.x] + scratch[384 + threadIdx.x]);
                    G.cluster_arrive_all();
                    G.cluster_wait_all();
                }
#pragma unroll 1
                for (int pc = 0; pc < 2; ++pc) {
                    const int j0 = col_of(pc) + (lane & 15);
                    float ty = 0.0f, f, gy;
                    if (i < LAST)
                        for (int q = 0; q < 4; ++q) ty += scratch[q * 128 + j0];
                    else
                        for (int r = 0; r < CL; ++r) ty += ws[tl.bred + (size_t)r * 128 + j0];
                    factors(i, i < LAST ? h0 + j0 : j0, j0 < col_lim(i), ty, q4 == 0 && lane < 16 && (i < LAST || rank == 0), f, gy);
                    ld_state(i, nxt + (size_t)i * dh, col_of(pc), y);
                    acc16(lanes + 128 * i + col_of(pc), t);
                    mask(i, col_of(pc), t);
#pragma unroll
                    for (int j = 0; j < 16; ++j) t[j] = __shfl_sync(0xffffffffu, f, j) * t[j] - y[j] * __shfl_sync(0xffffffffu, gy, j);
                    acc_st16(lanes + 128 * i + col_of(pc), t);
                    put(true, 0, i, col_of(pc), t);
                }
                G.epi_sync();
            }
            tmem_wait_st();
            G.signal(&sh.ops);
        }

        // The carries' adjoints <T, W>, <T, M>, <S, M>; T <- cw T, S <- cm T + cb S, while the first products run.  The next piece's W, M
        // are under way while this one's S is written (L1, what is left of it, holds 28 KB of loads in flight)
        {
            float pw = 0.0f, pm = 0.0f, pb = 0.0f, w[16], m[16];
            auto ld_wm = [&](int e) {
                ld_raw(e >> 1, ck + (size_t)(e >> 1) * dh, col_of(e & 1), w);
                ld_raw(e >> 1, ck + (size_t)(NMAT + (e >> 1)) * dh, col_of(e & 1), m);
            };
            const float cw = sc.cw, cm = sc.cm, cb = sc.cb;
            ld_wm(0);
#pragma unroll 1
            for (int e = 0; e < 2 * NMAT; ++e) {
                const int i = e >> 1, col = col_of(e & 1);
                float t[16], sv[16];
                ld_raw(i, ws + lay.S[i], col, sv);
                mask(i, col, w);
                mask(i, col, m);
                acc16(lanes + 128 * i + col, t);
                mask(i, col, t);  // lanes past the matrix collect whatever the MMAs read past the operands
#pragma unroll
                for (int j = 0; j < 16; ++j) { pw += t[j] * w[j]; pm += t[j] * m[j]; }
                mask(i, col, sv);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    pb += sv[j] * m[j];
                    sv[j] = cm * t[j] + cb * sv[j];
                    t[j] *= cw;
                }
                acc_st16(lanes + 128 * i + col, t);
                if (e + 1 < 2 * NMAT) ld_wm(e + 1);
                st_state(i, ws + lay.S[i], col, sv);
                put(false, buf ^ 1, i, col, sv);
            }
            tmem_wait_st();
            pw = warp_sum(pw); pm = warp_sum(pm); pb = warp_sum(pb);
            if (lane == 0) { sh.dots[n & 1][warp][0] = pw; sh.dots[n & 1][warp][1] = pm; sh.dots[n & 1][warp][2] = pb; }
            G.signal(&sh.scaled);
        }

        // ---- everything that meets (T, S) directly.  G_t enters W_C with K^W_t and M_C with K^M_t: its adjoint is K^W_t T + K^M_t S
#pragma unroll 1
        for (int tk = 0; tk < tbn; ++tk) {
            float kwb = 0.0f, kmb = 0.0f;  // adjoints of K^W, K^M of token 16 grp + (lane >> 1): this warp's lanes
            float* kb = sh.kb[warp];
            float c1[16], c2[16], z0[16], z1[16];
            const size_t e0 = (((size_t)(on_h ? bl : b0) * tb + tk) * 64 + 16 * grp) * 64 + (row & 63);
            auto ld_col = [&](size_t src, float (&v)[16]) {
                const float* p = sl + src + e0;
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = p[64 * j];
            };
            {
                const int t = tk * 64 + 16 * grp + (lane & 15);
                __syncwarp();
                kb[lane] = t < len ? (lane < 16 ? sc.kW[t] : sc.kM[t]) : 0.0f;
                __syncwarp();
            }
            auto no_h = [&](float (&x)[16], float (&y)[16]) {  // lanes without a hidden unit hold whatever the MMA read
                if (!on_h)
#pragma unroll
                    for (int j = 0; j < 16; ++j) x[j] = y[j] = 0.0f;
            };
            // x = T_first k, y = S_first k: adjoint of pz; through pz = ph act'(z) to phb and the second-order part of zb
            {
                float phb[16], ph[16], g1[16];
                ld_col(tl.sph, ph);
                ld_col(tl.sc1, c1);
                ld_col(tl.sc4, z0);
                if (SW) ld_col(tl.sg1, g1);
                G.job_out([&](uint32_t t) {
                    float x[16], y[16];
                    acc16(t + 16 * grp, x);
                    acc16(t + 64 + 16 * grp, y);
                    no_h(x, y);
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float pz = ph[j] * c1[j], pzb = -(kb[j] * x[j] + kb[16 + j] * y[j]);
                        x[j] *= pz;
                        y[j] *= pz;
                        phb[j] = pzb * c1[j];
                        z0[j] *= pzb;
                        if (SW) { g1[j] *= ph[j]; z1[j] = pzb * g1[j]; }
                    }
                    kwb -= reduce16(x, lane);
                    kmb -= reduce16(y, lane);
                });
                if constexpr (SW) {
                    ld_col(tl.sc2, c2);
                    G.job_out([&](uint32_t t) {
                        float x[16], y[16];
                        acc16(t + 16 * grp, x);
                        acc16(t + 64 + 16 * grp, y);
                        no_h(x, y);
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const float pz = ph[j] * c2[j], pzb = -(kb[j] * x[j] + kb[16 + j] * y[j]);
                            x[j] *= pz;
                            y[j] *= pz;
                            phb[j] += pzb * c2[j];
                            z0[j] += pzb * g1[j];
                        }
                        kwb -= reduce16(x, lane);
                        kmb -= reduce16(y, lane);
                    });
                }
                if (on_h) st_split16(blk(tl.bPhb) + ((size_t)bl * tb + tk) * B, row & 63, 16 * grp, phb);
                if (tk == tbn - 1) G.signal(&sh.phb);
            }
            // T_last^T pu = x, S_last^T pu = y: adjoint of the activation through the last matrix's aggregation, -(K^W x + K^M y)
            G.job_out([&](uint32_t t) {
                float x[16], y[16];
                acc16(t + 16 * grp, x);
                acc16(t + 64 + 16 * grp, y);
                if (!on_h) return;
                float* o0 = ws + tl.bz0[0] + e0;
                float* o1 = ws + tl.bz0[LAST - 1] + e0;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float ab = -(kb[j] * x[j] + kb[16 + j] * y[j]);
                    o0[64 * j] = z0[j] + ab * c1[j];
                    if (SW) o1[64 * j] = z1[j] + ab * c2[j];
                }
            });
            float pv[16];
            {
                const float* p = sl + tl.spu + (size_t)(tk * 64 + 16 * grp) * dp + min(row, dp - 1);
                const int nt = len - tk * 64 - 16 * grp, ld = opaque(dp);
#pragma unroll
                for (int j = 0; j < 16; ++j, p += ld) pv[j] = *p;
#pragma unroll
                for (int j = 0; j < 16; ++j) pv[j] = row < dp && j < nt ? pv[j] : 0.0f;
            }
            // share of pub = -(K^W T_last a + K^M S_last a) + ..; with pu: the last matrix's part of the adjoints of K^W, K^M
            G.job_out([&](uint32_t t) {
                float x[16], y[16];
                acc16(t + 16 * grp, x);
                acc16(t + 64 + 16 * grp, y);
                float* out = partial(tl.bslot, 0, tk);
                const int ld = opaque(dp);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    if (row < dp) *out = -(kb[j] * x[j] + kb[16 + j] * y[j]);
                    out += ld;
                    x[j] = row < dp ? x[j] * pv[j] : 0.0f;
                    y[j] = row < dp ? y[j] * pv[j] : 0.0f;
                }
                kwb -= reduce16(x, lane);
                kmb -= reduce16(y, lane);
            });
            if ((lane & 1) == 0) {  // the gate kernel adds the shares up
                float* o = sl + tl.skwb + (size_t)(4 * rank + q4) * tb * 64 + tk * 64 + 16 * grp + (lane >> 1);
                o[0] = kwb;
                o[(size_t)kTileShares * tb * 64] = kmb;
            }
            // share of dk = -(K^W T_first^T pz + K^M S_first^T pz) + ..
            G.job_out([&](uint32_t t) {
                float x[16], y[16];
                acc16(t + 16 * grp, x);
                acc16(t + 64 + 16 * grp, y);
                float* out = partial(tl.bdk[buf], 0, tk);
                const int ld = opaque(dp);
                if (row < dp)
#pragma unroll
                    for (int j = 0; j < 16; ++j, out += ld) *out = -(kb[j] * x[j] + kb[16 + j] * y[j]);
            });
        }
        auto plain_share = [&](size_t base) {
#pragma unroll 1
            for (int tk = 0; tk < tbn; ++tk)
                G.job_out([&](uint32_t t) {
                    float x[16];
                    acc16(t + 16 * grp, x);
                    float* out = partial(base, 1, tk);
                    const int ld = opaque(dp);
                    if (row < dp)
#pragma unroll
                        for (int j = 0; j < 16; ++j, out += ld) *out = x[j];
                });
        };
        plain_share(tl.bslot);  // pub += W_last phb
        G.cluster_arrive_all();

        G.cluster_wait_all();

        // ---- rows, dealt to the cluster's warps.  Warps 0-7: pu = J(u) e, e = k + y - v, y = LN(u): adjoints of e and u; dv.
        // Warps 8-15: dk of the chunk before
        if (warp < 8) {
            for (int t = rank * 8 + warp; t < tbn * 64; t += CL * 8) {
                float ub[4] = {0.f, 0.f, 0.f, 0.f};
                if (t < len) {
                    float pub[4] = {0.f, 0.f, 0.f, 0.f}, y[4] = {0.f, 0.f, 0.f, 0.f}, pw[4] = {0.f, 0.f, 0.f, 0.f}, eb[4], ng[4];
                    const float r = sl[tl.sr + t], mey = sl[tl.smey + t], inv = 1.0f / (float)d;
                    if (ci < dp) {
                        const float4 y4 = *reinterpret_cast<const float4*>(sl + tl.sy + (size_t)t * dp + ci);
                        const float4 p4 = *reinterpret_cast<const float4*>(sl + tl.spu + (size_t)t * dp + ci);
                        add_parts<8>(ws + tl.bslot + (size_t)t * dp + ci, 2 * CL, (size_t)tb * 64 * dp, pub);
                        y[0] = y4.x; y[1] = y4.y; y[2] = y4.z; y[3] = y4.w;
                        pw[0] = p4.x; pw[1] = p4.y; pw[2] = p4.z; pw[3] = p4.w;
                    }
                    const float sx = warp_sum(sum4(pub)) * inv, mpy = warp_sum(dot4(pub, y)) * inv, spp = warp_sum(dot4(pub, pw));
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        eb[j] = ci + j < d ? r * (pub[j] - sx - y[j] * mpy) : 0.0f;
                        ng[j] = -eb[j];
                    }
                    const float s2 = warp_sum(sum4(eb)) * inv, s2y = warp_sum(dot4(eb, y)) * inv;
                    // second-order term of the LN Jacobian, and dy -> du for the y inside e
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        ub[j] = ci + j < d ? r * (eb[j] - s2 - y[j] * s2y) - r * inv * spp * y[j] - r * (mpy * pw[j] + mey * eb[j]) : 0.0f;
                    st_tok4(reinterpret_cast<__nv_bfloat16*>(a.dv) + ((size_t)seq * a.Ls + s + t) * d, ci, d, ng);
                    if (ci < dp) *reinterpret_cast<float4*>(ws + tl.bEb[buf] + (size_t)t * dp + ci) = make_float4(eb[0], eb[1], eb[2], eb[3]);
                }
                if (ci < dp) st_split4<true>(blk(tl.bUk) + (size_t)((t >> 6) * db + (lane >> 4)) * B, t & 63, ci & 63, ub);
            }
        } else if (g + 1 < ga.ng) {
            const int s1 = s + a.C, len1 = min(a.C, a.L - s1);
            for (int t = rank * 8 + warp - 8; t < len1; t += CL * 8) dk_row(s1, t, buf ^ 1);
        }
        G.cluster_arrive_all();

        // A product's contribution to T of matrix i, rounded to nearest onto the master; `done`: the last one, T's operand blocks follow.
        // Accumulated onto the master itself, every MMA truncated T, chunk after chunk: 64 chunks of 64 tokens, d = 128, h = 512, error
        // of the adjoints against 64 bits 3.1e-5 (first matrix) and 3.3e-5 (momentum of the last), this way 9.8e-6 and 7.0e-6; the
        // step takes as long (15.2 ms for 64 sequences)
        auto contribution = [&](int i, bool done) {
            G.job_out([&](uint32_t t) {
#pragma unroll 1
                for (int pc = 0; pc < 2; ++pc) {
                    const int col = col_of(pc);
                    float x[16], m[16];
                    acc16(t + col, x);
                    acc16(lanes + 128 * i + col, m);
#pragma unroll
                    for (int j = 0; j < 16; ++j) m[j] += x[j];
                    acc_st16(lanes + 128 * i + col, m);
                    if (done && !NORMED) {
                        mask(i, col, m);
                        put(true, 0, i, col, m);
                    }
                }
                tmem_wait_st();
            });
        };
#pragma unroll 1
        for (int k = 0; k < EARLY; ++k) contribution(min(k, LAST), false);

        // ---- u = W_last a ; a = act(z): adjoint of z
#pragma unroll 1
        for (int tk = 0; tk < tbn; ++tk) {
            const size_t e0 = (((size_t)(on_h ? bl : b0) * tb + tk) * 64 + 16 * grp) * 64 + (row & 63);
            float z0[16], z1[16], c1[16], c2[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                z0[j] = ws[tl.bz0[0] + e0 + 64 * j];
                c1[j] = sl[tl.sc1 + e0 + 64 * j];
                if (SW) {
                    z1[j] = ws[tl.bz0[LAST - 1] + e0 + 64 * j];
                    c2[j] = sl[tl.sc2 + e0 + 64 * j];
                }
            }
            if (tk == 0) G.cluster_wait_all();
            G.job_out([&](uint32_t t) {
                float x[16];
                acc16(t + 16 * grp, x);
                if (!on_h) return;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    z0[j] += x[j] * c1[j];
                    if (SW) z1[j] += x[j] * c2[j];
                }
                st_split16(blk(tl.bZk[0]) + ((size_t)bl * tb + tk) * B, row & 63, 16 * grp, z0);
                if (SW) st_split16(blk(tl.bZk[LAST - 1]) + ((size_t)bl * tb + tk) * B, row & 63, 16 * grp, z1);
            });
        }
        G.signal(&sh.zb);
#pragma unroll 1
        for (int k = EARLY; k < LAST + 3; ++k) contribution(min(k, LAST), k == LAST + 2);
        plain_share(tl.bdk[buf]);  // dk += W_first^T zb
#pragma unroll 1
        for (int i = 0; i < LAST; ++i) contribution(i, true);

        if (warp == 0) {
            G.await(&sh.scaled, n, 409);  // every warp's share of the dot products
            if (lane < 3) {
                float x = 0.0f;
                for (int w = 0; w < 16; ++w) x += sh.dots[n & 1][w][lane];
                sl[tl.sdots + rank * 4 + lane] = x;
            }
        }
        if (!NORMED) G.signal(&sh.ops);
    }
    G.cluster_arrive_all();
    G.cluster_wait_all();
    {
        const int s = ga.c0 * a.C, len = min(a.C, a.L - s);
        for (int t = rank * 16 + warp; t < len; t += CL * 16) dk_row(s, t, ga.c0 & 1);
        const bool out = ga.last && !a.carry_out;
#pragma unroll 1
        for (int e = 0; e < 2 * NMAT; ++e) {
            const int i = e >> 1, col = col_of(e & 1);
            float t[16];
            acc16(lanes + 128 * i + col, t);
            st_state(i, out ? a.dW_init[i] + (size_t)seq * dh : ws + lay.T[i], col, t);
            if (out) {
                ld_state(i, ws + lay.S[i], col, t);
                st_state(i, a.dM_init[i] + (size_t)seq * dh, col, t);
            }
        }
    }
    G.teardown();
}

template <int KIND, bool NORMED, bool BESIDE> int launch(const GroupArgs& ga, const NextGroup& next, int rec_ctas, cudaStream_t st) {
    static bool attr_done[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return (int)cudaGetLastError();
    if (dev < 0 || dev >= 64 || !attr_done[dev]) {
        cudaError_t e = cudaFuncSetAttribute(tile_chain_kernel<KIND, NORMED, BESIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kChainSmem);
        if (e != cudaSuccess) return (int)e;
        if (dev >= 0 && dev < 64) attr_done[dev] = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(ga.a.N * ga.a.cl + rec_ctas));
    cfg.blockDim = dim3(chain_threads(KIND));
    cfg.dynamicSmemBytes = kChainSmem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)ga.a.cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, tile_chain_kernel<KIND, NORMED, BESIDE>, ga, next);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaGetLastError();
}

}  // namespace

int tile_chain_launch(const tile::GroupArgs& ga, const tile::NextGroup& next, int rec_ctas, int kind, cudaStream_t st) {
    auto go = [&](auto kind_, auto normed) {
        return rec_ctas > 0 ? launch<decltype(kind_)::value, decltype(normed)::value, true>(ga, next, rec_ctas, st)
                            : launch<decltype(kind_)::value, decltype(normed)::value, false>(ga, next, 0, st);
    };
    using std::integral_constant;
    if (ga.a.row_norm[0]) return kind == 0 ? go(integral_constant<int, 0>(), std::true_type()) : go(integral_constant<int, 1>(), std::true_type());
    return kind == 0 ? go(integral_constant<int, 0>(), std::false_type()) : go(integral_constant<int, 1>(), std::false_type());
}

}  // namespace e2ttt
