// Tensor-core base-case block product for sm_103a (Sec. 3.10 inner layer,
// re-designed for tcgen05): C = A * Bt^T over GF(2) or the Boolean algebra,
// A (m x k) and Bt (n x k) packed along k.
//
// The bit product is an integer dot product of 0/1 vectors: count_ij =
// sum_k A_ik Bt_jk. GF(2) takes count mod 2, Boolean takes count > 0. The
// tensor cores compute the counts exactly: bits are expanded to e4m3 bytes
// (value 2^-6, products 2^-12, FP32 accumulation exact while counts stay
// below 2^23). sm_103a has no 8-bit integer MMA (ptxas rejects
// tcgen05.mma kind::i8 for this target), so FP8 is the exact tensor format.
//
// Persistent kernel, one CTA per SM, warp-specialised (18 warps):
//   warp 16     TMA producer: packed tiles of 128 rows of A and 256 rows of
//               Bt (128 in a pair, below), 256 bits of k each (32-byte rows),
//               into a PSTAGES-deep shared ring (cp.async.bulk.tensor,
//               mbarrier complete_tx). Each packed stage feeds two operand
//               stages of 128 bits.
//   Bt expansion (8 warps; 4 in a pair): each packed 32-bit word becomes
//               32 bytes of the K-major, 128-byte-swizzled canonical UMMA
//               layout; a warp expands 4 whole rows of a packed stage at a
//               time.
//   A expansion (4 warps, one per TMEM lane quarter): one row per thread,
//               every packed stage: 256 bits -> 256 e4m3 bytes (both operand
//               stages) written straight into TMEM with one tcgen05.st.
//   epilogue (4 warps; 8 in a pair, two per lane quarter splitting the
//               columns): tcgen05.ld 32 lanes x 32 columns at a time, parity
//               or non-zero test, bits packed in registers with a shallow
//               tree (one row per thread) and stored as 64-bit words.
//   warp 17     MMA issuer: per packed stage, 2 x 4 tcgen05.mma (M=128,
//               N=256, K=32; A from TMEM, B from shared memory) into the TMEM
//               accumulator and one commit that frees the operand slot.
// SM pairs (PAIR): two CTAs of a cluster on two SMs share one 256 x 256 tile
// through tcgen05.mma.cta_group::2 (M=256). Each CTA expands its own 128 rows
// of A into its TMEM and its own 128 of the tile's 256 Bt rows into its
// shared memory; the even CTA issues the MMAs, which read both CTAs'
// operands and accumulate each CTA's 128 rows in its own TMEM. The gating
// barriers (operand stage full, accumulator empty) live in the even CTA and
// both CTAs' producers and epilogues arrive there; the commits that free an
// operand stage or publish the accumulator are multicast to both CTAs.
// The two operand stages a packed stage fills form one slot with one "full"
// barrier (every producer arrives) and one "empty" barrier (one commit).
// Every producer handles every packed stage in order, so the MMA issuer's
// wait on a slot covers the slots before it too: with four or more slots it
// checks one barrier per two packed stages (a check costs ~190 cycles of
// latency, even when the phase is already complete). TMEM stores share the tensor pipe's issue path
// with the MMAs, so A goes in with one wide store per packed stage. Keeping
// A in TMEM means shared memory carries only Bt (written once, read once by
// the tensor core). Long k is flushed from TMEM in chunks of `kchunk` stages
// (the epilogue folds parities / ORs across chunks).
//
// Within every 32-element group of k the expansion permutes k (byte t of
// output word j holds bit 8t + j of the packed word); A and Bt use the same
// permutation, so the contraction is unchanged.
//
// In-kernel level (LEVEL, SM pairs): e2m1 operands, every bit a 4-bit value
// under a uniform block scale, twice the k per MMA (kind::mxf4, K = 64); an
// operand stage then holds 256 bits of k and a packed stage 512. (The e2m1
// base case itself is tc_fp4.cu.)
//
// Batched form (BATCHED): each unit walks its own list of work items, one
// tile of one problem each (per-problem TMA maps); a tile may run N = 128
// MMAs (a tail with at most 128 columns inside n) and may end in half a
// packed stage. Uniform form: the tiles of `count` equal leaves.
//
// Every mbarrier wait is bounded (wall clock, ~2 s). A wait that gives up
// records BMM device error DEVERR_TIMEOUT and makes its role stop; the CTA
// then drains its own in-flight copies and MMAs (again bounded), frees TMEM
// and returns.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cstring>
#include <mutex>

#include "plan.h"
#include "tc_batched.h"
#include "tc_ptx.cuh"

namespace bmm {
namespace {

constexpr int BM = TC_TILE_M;    // rows of C per tile (UMMA M, TMEM lanes)
constexpr int SUB = 2;           // operand stages per packed stage
constexpr int KS_MIN = 128;      // k granularity of the operands (both formats)
// 18 warps: an SM sub-partition (16 K registers) holds at most five of
// them, which leaves 96 registers per thread (the A expansion keeps 64
// output words live for one wide TMEM store). Warps 0..15 are split between
// Bt expansion, A expansion (one warp per TMEM lane quarter) and the
// epilogue as the layout below gives; then the TMA and MMA warps.
constexpr int AEXP_WARPS = 4;
constexpr int TMA_WARP = 16;
constexpr int MMA_WARP = 17;
constexpr int THREADS = 18 * 32;

// An operand stage is 128 bytes of expanded operand per row in both
// formats: 128 k as e4m3 bytes, or 256 k as e2m1 nibbles (two per byte).
// One tcgen05.mma consumes 32 bytes of k per row (K = 32 e4m3, K = 64 e2m1),
// so the descriptors and TMEM columns advance the same way in both.
constexpr int ACC_COL = 0;               // accumulator: TMEM columns [0, BN)
constexpr int A_COL = BN;                // A ring: columns [BN, BN + ESTAGES * A_STAGE_COLS)
constexpr int A_STAGE_COLS = 32;         // 128 bytes of a row = 32 columns of 32 bits
constexpr int A_MMA_COLS = 8;            // 32 bytes of a row per MMA
constexpr int MMAS_PER_STAGE = 4;
constexpr int SF_COL = 448;              // e2m1: block scales, columns [448, 512)
constexpr int SF_COLS = 64;

// Per-CTA shapes and shared-memory layout. A CTA always owns 128 rows of C
// (its 128 TMEM lanes) and the matching 128 rows of A. A CTA on its own
// (cta_group::1) also expands all 256 Bt rows of its 128 x 256 tile. In a
// pair (a cluster of two CTAs on two SMs, cta_group::2, one 256 x 256 tile)
// each CTA expands only its half of the Bt rows, and the pair's MMAs read
// both halves: per SM, half the shared-memory traffic and a third less
// expansion work for the same number of MACs.
// LEVEL: the in-kernel Strassen level (below). Its packed stages hold up to
// six quadrant tiles (the A quadrants one product combines, then its Bt
// quadrants; at most six for every variant's products), so the ring is two
// packed stages deep.
template <bool PAIR, bool LEVEL = false>
struct Lay {
    static constexpr bool FP4 = LEVEL;
    static constexpr int KS = FP4 ? 256 : 128;  // k (bits) per operand stage
    static constexpr int KP = SUB * KS;         // k (bits) per packed (TMA) stage
    static constexpr int MMA_K = FP4 ? 64 : 32; // k per tcgen05.mma
    // ring depths: packed stages (shared) and operand stages (Bt in shared,
    // A in TMEM); a pair's smaller operand stages leave room for deeper rings.
    // The e2m1 form gives up two operand stages of TMEM to the block scales.
    static constexpr int PSTAGES = LEVEL ? 2 : PAIR ? 6 : 4;
    static constexpr int ESTAGES = PAIR ? (FP4 ? 6 : 8) : 4;
    // operand slots: the two operand stages one packed stage fills
    static constexpr int OSLOTS = ESTAGES / SUB;
    // packed stages the MMA issuer covers with one wait (needs more slots
    // than that, or the producers cannot run ahead)
    static constexpr int WAITG = OSLOTS >= 4 ? 2 : 1;
    // barriers: full_p[P], empty_p[P], full_o[O], empty_o[O], acc_full, acc_empty, drain
    static constexpr int NBARS = 2 * PSTAGES + 2 * OSLOTS + 3;
    // warps: Bt expansion [0, BEXP_WARPS), A expansion [AEXP_WARP0, +4),
    // epilogue [EPI_WARP0, TMA_WARP). A CTA alone has twice the Bt rows, a
    // pair's MMA issuer gains most from a short accumulator drain.
    static constexpr int BEXP_WARPS = PAIR ? 4 : 8;
    static constexpr int AEXP_WARP0 = BEXP_WARPS;
    static constexpr int EPI_WARP0 = AEXP_WARP0 + AEXP_WARPS;
    static constexpr int EPI_WARPS = TMA_WARP - EPI_WARP0;
    static_assert(AEXP_WARP0 % 4 == 0 && EPI_WARP0 % 4 == 0 && EPI_WARPS % 4 == 0,
                  "warp % 4 is the TMEM lane quarter");
    static constexpr int TILE_M = PAIR ? 2 * BM : BM;  // rows of C per tile
    static constexpr int BROWS = PAIR ? BN / 2 : BN;   // Bt rows held by one CTA
    static constexpr int PA_BYTES = BM * KP / 8;       // packed A per packed stage
    static constexpr int PB_BYTES = BROWS * KP / 8;    // packed Bt per packed stage
    static constexpr int EB_BYTES = BROWS * 128;       // expanded Bt per operand stage
    static constexpr int QTILES = 6;                   // LEVEL: quadrant tiles per stage
    static constexpr int OFF_EB = 0;
    static constexpr int OFF_PA = OFF_EB + ESTAGES * EB_BYTES;
    static constexpr int OFF_PB = OFF_PA + PSTAGES * PA_BYTES;  // (not LEVEL)
    static constexpr int PSTAGE_BYTES = QTILES * PA_BYTES;      // LEVEL: one packed stage
    // LEVEL: every epilogue thread's words of the four C quadrants (4 x 4
    // words, lane-interleaved), in shared memory beside the registers the
    // accumulator loads need
    static constexpr int QOUT_BYTES = LEVEL ? EPI_WARPS * 32 * 16 * 4 : 0;
    static constexpr int OFF_QOUT = LEVEL ? OFF_PA + PSTAGES * PSTAGE_BYTES : 0;
    // batched: two work items per epilogue warp, fetched a tile ahead
    static constexpr int OFF_ITEMS = LEVEL ? OFF_QOUT + QOUT_BYTES : OFF_PB + PSTAGES * PB_BYTES;
    static constexpr int ITEM_BYTES = 48;
    static constexpr int OFF_BAR = OFF_ITEMS + EPI_WARPS * 2 * ITEM_BYTES;
    static constexpr int OFF_TMEM_SLOT = OFF_BAR + NBARS * 8;
    static constexpr int SMEM_BYTES = OFF_TMEM_SLOT + 16 + 1024;  // + alignment slack
    static_assert(EB_BYTES % 1024 == 0, "swizzle atoms stay 1024-byte aligned");
    static_assert(A_COL + ESTAGES * A_STAGE_COLS <= (FP4 ? SF_COL : TMEM_COLS), "TMEM budget");
    static_assert(SF_COL + SF_COLS <= TMEM_COLS, "TMEM budget");
    static_assert(KS / MMA_K == MMAS_PER_STAGE && MMA_K * (FP4 ? 4 : 8) == 32 * A_MMA_COLS,
                  "an MMA reads 32 bytes of k per row");
    static_assert(ESTAGES % SUB == 0, "a packed stage's operand stages are adjacent in TMEM");
    static_assert(SMEM_BYTES <= 227 * 1024, "shared memory budget");
    static_assert(!LEVEL || (PAIR && PA_BYTES == PB_BYTES), "LEVEL: equal quadrant tiles");
};

// Self-test of the bounded wait: one thread waits on a barrier that nothing
// arrives on, gives up after limit_ns, records the timeout and returns.
__global__ void wait_selftest_kernel(uint32_t* err, uint64_t limit_ns) {
    __shared__ __align__(8) uint64_t bar;
    const uint32_t b = smem_u32(&bar);
    mbar_init(b, 1);
    fence_barrier_init();
    mbar_wait_slow(b, 0, err, limit_ns);
}

struct Params {
    // uniform form: one shape, `count` leaves side by side
    uint64_t* C;
    int64_t ldc, strideC;
    int m, n, nks, op;
    int tiles_m, tiles_n, total_tiles;
    // batched form: per-problem descriptors and per-CTA work lists
    const TcProblem* probs;
    const TcWorkItem* items;
    const int32_t* cta_ptr;
    int kchunk;  // stages per flush (both forms)
    uint32_t* err;
    Spread sp;
    // LEVEL: each leaf is a block of 2m x 2k times 2k x 2n bits whose seven
    // quadrant products run here (m, n, nks: one quadrant product); qkw:
    // words of k per quadrant; nibble h of xi4 / eta4: the A / B quadrants
    // product h combines; bits 7q..7q+6 of zeta7: the products C quadrant q
    // sums.
    uint32_t xi4, eta4, zeta7;
    int qkw;
};

// Everything a role needs about one output tile.
struct Tile {
    const CUtensorMap* ma;
    const CUtensorMap* mb;
    uint64_t* C;  // leaf's C
    int64_t ldc;
    int m, n, nks, op, tm, tn, leaf;
    int n128;     // batched: N = 128 MMAs (columns 128.. of the tile lie past n)
};

// Scheduling unit: a CTA, or a CTA pair (consecutive blockIdx.x, one cluster).
template <bool PAIR>
__device__ __forceinline__ int unit_id() {
    return PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
}
template <bool PAIR>
__device__ __forceinline__ int unit_count() {
    return PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
}

template <bool BATCHED, bool PAIR>
__device__ __forceinline__ int tile_count(const Params& p) {
    const int u = unit_id<PAIR>();
    if (BATCHED) return p.cta_ptr[u + 1] - p.cta_ptr[u];
    int c = 0;
    for (int t = u; t < p.total_tiles; t += unit_count<PAIR>()) c++;
    return c;
}

// A batched tile from its work item.
__device__ __forceinline__ Tile tile_of_item(const Params& p, const TcWorkItem& w) {
    Tile t;
    const TcProblem* d = p.probs + w.prob;
    t.ma = &d->mapA;
    t.mb = &d->mapB;
    t.C = w.C;
    t.ldc = w.ldc;
    t.m = w.m;
    t.n = w.n;
    t.nks = w.nks;
    t.op = w.op;
    t.tm = w.tm;
    t.tn = w.tn;
    t.leaf = 0;
    t.n128 = w.n128;
    return t;
}

// items: batched, this unit's slice of the work list (read once per kernel,
// so that fetching a tile's item is one load, not two dependent ones).
template <bool BATCHED, bool PAIR>
__device__ __forceinline__ Tile tile_get(const Params& p, const TcWorkItem* items, int idx,
                                         const CUtensorMap* tmA, const CUtensorMap* tmB) {
    Tile t;
    if (BATCHED) {
        const TcWorkItem w = items[idx];
        const TcProblem* d = p.probs + w.prob;
        t.ma = &d->mapA;
        t.mb = &d->mapB;
        t.C = w.C;
        t.ldc = w.ldc;
        t.m = w.m;
        t.n = w.n;
        t.nks = w.nks;
        t.op = w.op;
        t.tm = w.tm;
        t.tn = w.tn;
        t.leaf = 0;
        t.n128 = w.n128;
    } else {
        const TileCoord c =
            tile_of(unit_id<PAIR>() + idx * unit_count<PAIR>(), p.tiles_m, p.tiles_n);
        t.ma = tmA;
        t.mb = tmB;
        t.C = p.C + (int64_t)c.leaf * p.strideC;
        t.ldc = p.ldc;
        t.m = p.m;
        t.n = p.n;
        t.nks = p.nks;
        t.op = p.op;
        t.tm = c.tm;
        t.tn = c.tn;
        t.leaf = c.leaf;
        t.n128 = 0;
    }
    return t;
}

// What the MMA issuer needs of a tile: its k stages, and (batched) N = 128.
struct TileK {
    int nks, n128;
};
template <bool BATCHED>
__device__ __forceinline__ TileK tile_k(const Params& p, const TcWorkItem* items, int idx) {
    if (BATCHED) {
        const TcWorkItem* w = items + idx;
        return {w->nks, w->n128};
    }
    return {p.nks, 0};
}

// The in-kernel Strassen level (LEVEL; a level shifted from the expanding
// and compressing passes into the inner layer, Sec. 3.15), binary product
// only: every leaf of the launch is a block of 2m x 2k times 2k x 2n bits,
// and a CTA pair takes one 256 x 256 tile position of the quadrant-sized
// product and runs the block's seven quadrant products there, one after the
// other. For product h the TMA producer loads, per packed stage, the tiles
// of the A quadrants that xi_h = alpha_h phi selects and of the Bt quadrants
// that eta_h = beta_h psi selects (the combined operators of Eqs. mb-* /
// ab-* / sw-*), the expansion warps XOR them as they expand, so the seven
// operands never exist in HBM, and the epilogue XORs the product's parity
// bits into the C quadrants that zeta = chi gamma sends it to, in
// registers; the four quadrant words of the position leave once, after the
// seventh product.
template <bool BATCHED, bool PAIR, bool LEVEL = false>
__global__ void __launch_bounds__(THREADS, 1)
    tc_nt_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const Params p) {
    static_assert(!LEVEL || (!BATCHED && PAIR), "the in-kernel level runs on SM pairs");
    using LY = Lay<PAIR, LEVEL>;
    constexpr bool FP4 = LEVEL;
    constexpr int PSTAGES = LY::PSTAGES, OSLOTS = LY::OSLOTS, KP = LY::KP;
    constexpr int BEXP_WARPS = LY::BEXP_WARPS, EPI_WARP0 = LY::EPI_WARP0,
                  EPI_WARPS = LY::EPI_WARPS;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = sbase + LY::OFF_BAR;
    auto full_p = [&](int s) { return bar0 + 8u * s; };
    auto empty_p = [&](int s) { return bar0 + 8u * (PSTAGES + s); };
    auto full_o = [&](int q) { return bar0 + 8u * (2 * PSTAGES + q); };
    auto empty_o = [&](int q) { return bar0 + 8u * (2 * PSTAGES + OSLOTS + q); };
    const uint32_t acc_full = bar0 + 8u * (2 * PSTAGES + 2 * OSLOTS);
    const uint32_t acc_empty = acc_full + 8u;
    const uint32_t drain_bar = acc_full + 16u;
    uint32_t* tmem_slot = (uint32_t*)(smem + LY::OFF_TMEM_SLOT);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // In a pair, CTA 0 issues the MMAs and holds the barriers that gate them
    // (full_o, acc_empty); both CTAs' producers and epilogues arrive there.
    const uint32_t rank = PAIR ? cluster_rank() : 0u;
    constexpr uint32_t CTAS = PAIR ? 2u : 1u;
    auto arrive_leader = [&](uint32_t bar) {
        if (PAIR)
            mbar_arrive_cluster(bar, 0);
        else
            mbar_arrive(bar);
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < PSTAGES; s++) {
            mbar_init(full_p(s), 1);
            mbar_init(empty_p(s), BEXP_WARPS + AEXP_WARPS);  // every expansion warp reads every stage
        }
        for (int q = 0; q < OSLOTS; q++) {
            mbar_init(full_o(q), CTAS * (BEXP_WARPS + AEXP_WARPS));
            mbar_init(empty_o(q), 1);
        }
        mbar_init(acc_full, 1);
        mbar_init(acc_empty, CTAS * EPI_WARPS);
        mbar_init(drain_bar, 1);
        fence_barrier_init();
    }
    if (warp == MMA_WARP) tmem_alloc<PAIR>(smem_u32(tmem_slot));
    if (!BATCHED && warp == TMA_WARP && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA))
                     : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB))
                     : "memory");
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync();  // the peer's barriers exist before anything arrives on them
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    const int kchunk = p.kchunk;
    const int my_tiles = tile_count<BATCHED, PAIR>(p);
    const TcWorkItem* my_items = BATCHED ? p.items + p.cta_ptr[unit_id<PAIR>()] : nullptr;
    int total_pit = 0;  // packed stages this CTA runs (batched: from the plan)
    if (BATCHED)
        total_pit = p.cta_ptr[unit_count<PAIR>() + 1 + unit_id<PAIR>()];
    else
        total_pit = my_tiles * (LEVEL ? 7 : 1) * (p.nks / SUB);
    // LEVEL: a packed stage's quadrant tiles, A's first (sub-buffer j)
    auto qtile = [&](int s, int j) {
        return (uint32_t)(LY::OFF_PA + s * LY::PSTAGE_BYTES + j * LY::PA_BYTES);
    };

    if (warp == TMA_WARP) {
        // ---------------------------------------------------- TMA producer
        if (lane == 0) {
            int pit = 0;  // packed stages issued
            bool ok = true;
            // Batched: a tile's work item is read two tiles ahead and its
            // TMA maps prefetched one tile ahead, so neither the item load
            // nor a map fetch stalls the copies of the tile before it.
            Tile nxt = my_tiles > 0 ? tile_get<BATCHED, PAIR>(p, my_items, 0, &tmA, &tmB) : Tile{};
            Tile nxt2 = my_tiles > 1 ? tile_get<BATCHED, PAIR>(p, my_items, 1, &tmA, &tmB) : nxt;
            if (BATCHED && my_tiles > 0) {
                prefetch_tensormap(nxt.ma);
                prefetch_tensormap(nxt.mb);
            }
            for (int i = 0; ok && i < my_tiles; i++) {
                const Tile tc = nxt;
                nxt = nxt2;
                if (BATCHED && i + 1 < my_tiles) {
                    prefetch_tensormap(nxt.ma);
                    prefetch_tensormap(nxt.mb);
                }
                if (i + 2 < my_tiles)
                    nxt2 = tile_get<BATCHED, PAIR>(p, my_items, i + 2, &tmA, &tmB);
                const int arow = tc.tm * LY::TILE_M + (int)rank * BM;
                // an N = 128 tile takes 64 of its columns from each CTA of a pair
                const int brow =
                    tc.tn * BN + (int)rank * (BATCHED && tc.n128 ? LY::BROWS / 2 : LY::BROWS);
                if (LEVEL) {
                    // A quadrant (r, c) at rows r m, words c qkw; B block (r, c)
                    // is stored transposed, as Bt rows c n, words r qkw
                    for (int h = 0; ok && h < 7; h++) {
                        const uint32_t xa = (p.xi4 >> (4 * h)) & 0xFu;
                        const uint32_t xb = (p.eta4 >> (4 * h)) & 0xFu;
                        const uint32_t bytes = (uint32_t)(__popc(xa) + __popc(xb)) * LY::PA_BYTES;
                        for (int kp = 0; kp < tc.nks / SUB; kp++, pit++) {
                            const int s = pit % PSTAGES;
                            if (!mbar_wait(empty_p(s), ((pit / PSTAGES) & 1) ^ 1, p.err)) {
                                ok = false;
                                break;
                            }
                            mbar_arrive_tx(full_p(s), bytes);
                            int j = 0;
                            for (int q = 0; q < 4; q++)
                                if ((xa >> q) & 1u)
                                    tma_load_3d(sbase + qtile(s, j++), tc.ma,
                                                (q & 1) * p.qkw + kp * (KP / 64),
                                                (q >> 1) * tc.m + arow, tc.leaf, full_p(s));
                            for (int q = 0; q < 4; q++)
                                if ((xb >> q) & 1u)
                                    tma_load_3d(sbase + qtile(s, j++), tc.mb,
                                                (q >> 1) * p.qkw + kp * (KP / 64),
                                                (q & 1) * tc.n + brow, tc.leaf, full_p(s));
                        }
                    }
                    continue;
                }
                for (int kp = 0; kp < (tc.nks + SUB - 1) / SUB; kp++, pit++) {
                    const int s = pit % PSTAGES;
                    if (!mbar_wait(empty_p(s), ((pit / PSTAGES) & 1) ^ 1, p.err)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_tx(full_p(s), LY::PA_BYTES + LY::PB_BYTES);
                    tma_load_3d(sbase + LY::OFF_PA + s * LY::PA_BYTES, tc.ma, kp * (KP / 64), arow,
                                tc.leaf, full_p(s));
                    tma_load_3d(sbase + LY::OFF_PB + s * LY::PB_BYTES, tc.mb, kp * (KP / 64), brow,
                                tc.leaf, full_p(s));
                }
            }
            // drain: the copies of the last issued stages must land before exit
            for (int j = 1; j <= PSTAGES && j <= pit; j++) {
                const int i = pit - j;
                if (!mbar_wait(full_p(i % PSTAGES), (i / PSTAGES) & 1, p.err)) break;
            }
        }
    } else if (LEVEL && warp < BEXP_WARPS) {
        // ---------------------------------------------------- Bt expansion, in-kernel level
        // Per packed stage: items of 2 rows x 16 packed words (both operand
        // stages). Lane = (half h, row rr of the item, word wl of the half):
        // word w = 8h + wl goes to 16-byte chunk wl of operand stage 2q + h.
        // A quarter-warp holds the 8 chunks of one row: 8 distinct bank groups.
        const int h = lane >> 4, rr = (lane >> 3) & 1, wl = lane & 7;
        const Spread sp = p.sp;
        int lv_k = 0, lv_h = 0;  // packed stage within the product, the product
        for (int pit = 0; pit < total_pit; pit++) {
            const int s = pit % PSTAGES;
            const int q = pit % OSLOTS;
            if (!mbar_wait(full_p(s), (pit / PSTAGES) & 1, p.err) ||
                !mbar_wait(empty_o(q), ((pit / OSLOTS) & 1) ^ 1, p.err))
                break;
            constexpr int ITEMS = (LY::BROWS / 2) / BEXP_WARPS;
            uint8_t* eb = smem + LY::OFF_EB + (2 * q + h) * LY::EB_BYTES;
            uint32_t x[ITEMS];
            // S_h: the XOR of the Bt quadrant tiles, stored after A's
            const int j0 = __popc((p.xi4 >> (4 * lv_h)) & 0xFu);
            const int nb = __popc((p.eta4 >> (4 * lv_h)) & 0xFu);
#pragma unroll
            for (int i = 0; i < ITEMS; i++) x[i] = 0u;
            for (int j = 0; j < nb; j++) {
                const uint32_t* pb = reinterpret_cast<const uint32_t*>(smem + qtile(s, j0 + j));
#pragma unroll
                for (int i = 0; i < ITEMS; i++)
                    x[i] ^= pb[((warp + BEXP_WARPS * i) * 2 + rr) * 16 + 8 * h + wl];
            }
            if (++lv_k == p.nks / SUB) {
                lv_k = 0;
                if (++lv_h == 7) lv_h = 0;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(empty_p(s));
#pragma unroll
            for (int i = 0; i < ITEMS; i++) {
                const int row = (warp + BEXP_WARPS * i) * 2 + rr;
                uint32_t y[4];
                spread4(x[i], sp, y);
                *reinterpret_cast<uint4*>(eb + row * 128 + ((wl ^ (row & 7)) * 16)) =
                    make_uint4(y[0], y[1], y[2], y[3]);
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) arrive_leader(full_o(q));
        }
    } else if (warp < BEXP_WARPS) {
        // ---------------------------------------------------- Bt expansion (shared)
        // Per packed stage: items of 4 rows x 8 packed words (both operand
        // stages). Lane = (half h, row rr of the item, word wl of the half):
        // word w = 4h + wl of the row goes to operand stage 2q + h of slot q.
        // A quarter-warp then holds two adjacent rows (opposite parity) x 4
        // words of one half, whose swizzled 16-byte chunks are 8 distinct bank
        // groups.
        const int h = lane >> 4, rr = (lane >> 2) & 3, wl = lane & 3;
        const Spread sp = p.sp;
        static_assert(SUB == 2, "a packed stage feeds two operand stages");
        for (int pit = 0; pit < total_pit; pit++) {
            const int s = pit % PSTAGES;
            const int q = pit % OSLOTS;
            if (!mbar_wait(full_p(s), (pit / PSTAGES) & 1, p.err) ||
                !mbar_wait(empty_o(q), ((pit / OSLOTS) & 1) ^ 1, p.err))
                break;
            constexpr int ITEMS = (LY::BROWS / 4) / BEXP_WARPS;
            const uint32_t* pb =
                reinterpret_cast<const uint32_t*>(smem + LY::OFF_PB + s * LY::PB_BYTES);
            uint8_t* eb = smem + LY::OFF_EB + (2 * q + h) * LY::EB_BYTES;
            uint32_t x[ITEMS];
#pragma unroll
            for (int i = 0; i < ITEMS; i++)
                x[i] = pb[((warp + BEXP_WARPS * i) * 4 + rr) * 8 + 4 * h + wl];
            __syncwarp();
            if (lane == 0) mbar_arrive(empty_p(s));
#pragma unroll
            for (int i = 0; i < ITEMS; i++) {
                const int row = (warp + BEXP_WARPS * i) * 4 + rr;
                uint8_t* rowp = eb + row * 128;
                uint32_t y[8];
                spread8(x[i], sp, y);
                *reinterpret_cast<uint4*>(rowp + (((2 * wl) ^ (row & 7)) * 16)) =
                    make_uint4(y[0], y[1], y[2], y[3]);
                *reinterpret_cast<uint4*>(rowp + (((2 * wl + 1) ^ (row & 7)) * 16)) =
                    make_uint4(y[4], y[5], y[6], y[7]);
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) arrive_leader(full_o(q));
        }
    } else if (warp < EPI_WARP0) {
        // ---------------------------------------------------- A expansion (TMEM)
        // One warp per TMEM lane quarter, one row per thread, every packed
        // stage: 256 bits -> 256 e4m3 bytes = both operand stages of the
        // slot, adjacent TMEM columns, one store.
        const int quarter = warp & 3;
        const int row = 32 * quarter + lane;
        const Spread sp = p.sp;
        const uint32_t tlane = (uint32_t)(32 * quarter) << 16;
        if (FP4) {
            // block scales for this lane quarter, before the first full_o arrive
            uint32_t f[64];
#pragma unroll
            for (int i = 0; i < 64; i++) f[i] = SCALE_WORD;
            tmem_st64(tmem + tlane + (uint32_t)SF_COL, f);
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        }
        int lv_k = 0, lv_h = 0;  // LEVEL: packed stage within the product, the product
        for (int pit = 0; pit < total_pit; pit++) {
            const int s = pit % PSTAGES;
            const int q = pit % OSLOTS;
            if (!mbar_wait(full_p(s), (pit / PSTAGES) & 1, p.err)) break;
            constexpr int NV = KP / 128;  // 16-byte vectors per packed row
            uint4 xv[NV];
            if (LEVEL) {
                // T_h: the XOR of the A quadrant tiles
                const int na = __popc((p.xi4 >> (4 * lv_h)) & 0xFu);
#pragma unroll
                for (int v = 0; v < NV; v++) xv[v] = make_uint4(0u, 0u, 0u, 0u);
                for (int j = 0; j < na; j++) {
                    const uint4* src =
                        reinterpret_cast<const uint4*>(smem + qtile(s, j) + row * (KP / 8));
#pragma unroll
                    for (int v = 0; v < NV; v++) {
                        const uint4 t = src[v];
                        xv[v].x ^= t.x;
                        xv[v].y ^= t.y;
                        xv[v].z ^= t.z;
                        xv[v].w ^= t.w;
                    }
                }
                if (++lv_k == p.nks / SUB) {
                    lv_k = 0;
                    if (++lv_h == 7) lv_h = 0;
                }
            } else {
                const uint4* src = reinterpret_cast<const uint4*>(smem + LY::OFF_PA +
                                                                  s * LY::PA_BYTES + row * (KP / 8));
#pragma unroll
                for (int v = 0; v < NV; v++) xv[v] = src[v];
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(empty_p(s));
            if (!mbar_wait(empty_o(q), ((pit / OSLOTS) & 1) ^ 1, p.err)) break;
            tc_fence_after();  // the slot's MMAs (seen complete) before our TMEM stores
            uint32_t y[64];
#pragma unroll
            for (int v = 0; v < NV; v++) {
                if (FP4) {
                    spread4(xv[v].x, sp, y + 16 * v);
                    spread4(xv[v].y, sp, y + 16 * v + 4);
                    spread4(xv[v].z, sp, y + 16 * v + 8);
                    spread4(xv[v].w, sp, y + 16 * v + 12);
                } else {
                    spread8(xv[v].x, sp, y + 32 * v);
                    spread8(xv[v].y, sp, y + 32 * v + 8);
                    spread8(xv[v].z, sp, y + 32 * v + 16);
                    spread8(xv[v].w, sp, y + 32 * v + 24);
                }
            }
            tmem_st64(tmem + tlane + (uint32_t)(A_COL + 2 * q * A_STAGE_COLS), y);
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_leader(full_o(q));
        }
    } else if (warp == MMA_WARP) {
        // ---------------------------------------------------- MMA issuer
        if (lane == 0 && rank == 0) {
            constexpr uint32_t idesc =
                FP4 ? instr_desc_mxf4<LY::TILE_M>() : instr_desc<LY::TILE_M>(1u);
            constexpr uint32_t idesc128 = FP4 ? instr_desc_mxf4<LY::TILE_M, BN / 2>()
                                              : instr_desc<LY::TILE_M, BN / 2>(1u);
            // operand stage e's descriptor: the start-address field (bytes >> 4)
            // moves by EB_BYTES >> 4 per stage; every stage lies below 256 KB,
            // so no carry
            const uint64_t db_base = smem_desc_sw128(sbase + LY::OFF_EB);
            // The issuing thread's own instructions sit on the tensor pipe's
            // critical path (one extra branch per stage measured 5 %), so the
            // slot and its phase are running counters, not divisions.
            static_assert(LY::WAITG == 1 || LY::WAITG == 2, "wait groups of one or two slots");
            int seg = 0, pit = 0;
            int q = 0;         // pit % OSLOTS
            uint32_t ph = 0;   // (pit / OSLOTS) & 1
            bool ok = true;
            // a tile's k stages are loaded one tile ahead (batched: from the
            // work list in global memory, off the issue path)
            // (batched: items read two tiles ahead of their use)
            TileK tk_next = my_tiles > 0 ? tile_k<BATCHED>(p, my_items, 0) : TileK{0, 0};
            TileK tk_next2 = my_tiles > 1 ? tile_k<BATCHED>(p, my_items, 1) : tk_next;
            // LEVEL: every tile position runs seven products, each an
            // accumulator tile of its own
            const int mma_tiles = LEVEL ? 7 * my_tiles : my_tiles;
            for (int i = 0; ok && i < mma_tiles; i++) {
                const int nks = tk_next.nks;
                const uint32_t id = BATCHED && tk_next.n128 ? idesc128 : idesc;
                tk_next = tk_next2;
                if (i + 2 < mma_tiles) tk_next2 = tile_k<BATCHED>(p, my_items, i + 2);
                int kin = 0;
                for (int ks = 0; ks < nks; ks += SUB, pit++) {
                    // Every producer fills the slots in order, so one wait on
                    // the last of WAITG consecutive slots covers them all. At a
                    // tile's first stage the operands are checked before the
                    // (longer) wait for the epilogue to free the accumulator.
                    const bool group = (pit & (LY::WAITG - 1)) == 0;
                    if (group) {
                        int qw = q;
                        uint32_t phw = ph;
                        if (LY::WAITG == 2 && pit + 1 < total_pit && ++qw == OSLOTS) {
                            qw = 0;
                            phw ^= 1u;
                        }
                        if (!mbar_wait(full_o(qw), phw, p.err)) {
                            ok = false;
                            break;
                        }
                    }
                    if (kin == 0) {
                        if (!mbar_wait(acc_empty, (seg & 1) ^ 1, p.err)) {
                            ok = false;
                            break;
                        }
                    }
                    if (group || kin == 0) tc_fence_after();
#pragma unroll
                    for (int sub = 0; sub < SUB; sub++) {
                        // batched: an odd k-stage count ends in half a packed
                        // stage, whose second operand stage is all padding
                        if (BATCHED && sub > 0 && ks + sub >= nks) break;
                        const int e = 2 * q + sub;
                        const uint32_t ta = tmem + (uint32_t)(A_COL + e * A_STAGE_COLS);
                        const uint64_t db = db_base + (uint64_t)(e * (LY::EB_BYTES >> 4));
#pragma unroll
                        for (int j = 0; j < MMAS_PER_STAGE; j++) {
                            const uint32_t acc = (kin > 0 || sub > 0 || j > 0) ? 1u : 0u;
                            if (FP4)
                                mma_f4_ta<PAIR>(tmem + ACC_COL, ta + j * A_MMA_COLS, db + 2 * j,
                                                BATCHED ? id : idesc, tmem + SF_COL,
                                                tmem + SF_COL + SF_COLS / 2, acc);
                            else
                                mma_f8_ta<PAIR>(tmem + ACC_COL, ta + j * A_MMA_COLS, db + 2 * j,
                                                BATCHED ? id : idesc, acc);
                        }
                    }
                    mma_commit<PAIR>(empty_o(q));
                    if (++q == OSLOTS) {
                        q = 0;
                        ph ^= 1u;
                    }
                    kin += SUB;
                    if (kin >= kchunk || ks + SUB >= nks) {
                        mma_commit<PAIR>(acc_full);
                        seg++;
                        kin = 0;
                    }
                }
            }
            if (!ok) {  // wait (bounded) for every MMA this thread issued
                mma_commit<PAIR>(drain_bar, 1);
                mbar_wait(drain_bar, 0, p.err);
            }
        }
    } else if (warp < TMA_WARP) {
        // ---------------------------------------------------- epilogue
        // EPI_WARPS / 4 warps per TMEM lane quarter, splitting the columns.
        const int quarter = warp & 3;  // TMEM lanes 32*quarter .. +31
        const int chalf = (warp - EPI_WARP0) >> 2;
        const uint32_t tlane = (uint32_t)(32 * quarter) << 16;
        constexpr int CW = BN / (EPI_WARPS / 4) / 32;  // 32-column chunks per warp
        int seg = 0;
        bool ok = true;
        // batched: each tile's work item is copied into this warp's shared
        // slot while the tile before it runs, off the accumulator hand-off path
        const uint32_t islot =
            sbase + (uint32_t)(LY::OFF_ITEMS + (warp - EPI_WARP0) * 2 * LY::ITEM_BYTES);
        static_assert(sizeof(TcWorkItem) == LY::ITEM_BYTES, "three 16-byte copies per item");
        auto fetch_item = [&](int idx) {
            if (lane < 3)
                cp_async16(islot + (uint32_t)((idx & 1) * LY::ITEM_BYTES + 16 * lane),
                           reinterpret_cast<const uint8_t*>(my_items + idx) + 16 * lane);
        };
        if (BATCHED && my_tiles > 0) fetch_item(0);
        for (int i = 0; ok && i < my_tiles; i++) {
            Tile tc;
            if (BATCHED) {
                cp_async_wait_all();
                __syncwarp();
                TcWorkItem w;
                std::memcpy(&w, smem + (islot - sbase) + (i & 1) * LY::ITEM_BYTES, sizeof(w));
                __syncwarp();
                if (i + 1 < my_tiles) fetch_item(i + 1);
                tc = tile_of_item(p, w);
            } else {
                tc = tile_get<BATCHED, PAIR>(p, my_items, i, &tmA, &tmB);
            }
            const int nseg = (tc.nks + kchunk - 1) / kchunk;
            const bool gf2 = tc.op == OP_GF2;
            // an N = 128 tile writes no accumulator column past 128: the warps
            // that drain those columns only hand the accumulator back
            const bool idle = BATCHED && PAIR && tc.n128 && chalf == 1;
            // LEVEL: this thread's words of the four C quadrants, summed over
            // the position's seven products: word (q, c) at qo[(CW q + c) 32]
            static_assert(!LEVEL || CW == 4, "four words per quadrant");
            uint32_t* qo = reinterpret_cast<uint32_t*>(smem + LY::OFF_QOUT) +
                           (warp - EPI_WARP0) * 32 * 16 + lane;
            if (LEVEL)
#pragma unroll
                for (int j = 0; j < 16; j++) qo[32 * j] = 0u;
            uint32_t out[1][CW];
#pragma unroll
            for (int c = 0; c < CW; c++) out[0][c] = 0u;
            for (int h = 0; ok && h < (LEVEL ? 7 : 1); h++) {
            // LEVEL: the C quadrants product h goes to (bit q)
            uint32_t zq = 0;
            if (LEVEL)
                for (int q = 0; q < 4; q++) zq |= ((p.zeta7 >> (7 * q + h)) & 1u) << q;
            uint32_t words[LEVEL ? 1 : CW];
#pragma unroll
            for (int c = 0; c < (LEVEL ? 1 : CW); c++) words[c] = 0u;
            for (int g = 0; g < nseg; g++, seg++) {
                if (!mbar_wait(acc_full, seg & 1, p.err)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                if (idle) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) arrive_leader(acc_empty);
                    continue;
                }
                if (LEVEL) {
                    // parities are XOR-linear: each chunk folds straight into
                    // the quadrants product h goes to
#pragma unroll
                    for (int c = 0; c < CW; c += 2) {
                        uint32_t v[64];
                        tmem_ld64(tmem + tlane + (uint32_t)(ACC_COL + 32 * (CW * chalf + c)), v);
                        if (c + 2 == CW) {
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) arrive_leader(acc_empty);
                        }
                        const uint32_t b0 = pack_bits<OP_GF2>(v), b1 = pack_bits<OP_GF2>(v + 32);
#pragma unroll
                        for (int q = 0; q < 4; q++)
                            if ((zq >> q) & 1u) {
                                qo[32 * (CW * q + c)] ^= b0;
                                qo[32 * (CW * q + c + 1)] ^= b1;
                            }
                    }
                    continue;
                }
                // 64 columns per load: half the load-wait round trips of 32
#pragma unroll
                for (int c = 0; c < CW; c += 2) {
                    uint32_t v[64];
                    tmem_ld64(tmem + tlane + (uint32_t)(ACC_COL + 32 * (CW * chalf + c)), v);
                    if (c + 2 == CW) {
                        // every column this warp drains is in registers: hand the
                        // accumulator back before packing the last chunk
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) arrive_leader(acc_empty);
                    }
                    if (gf2) {
                        words[c] ^= pack_bits<OP_GF2>(v);
                        words[c + 1] ^= pack_bits<OP_GF2>(v + 32);
                    } else {
                        words[c] |= pack_bits<OP_BOOL>(v);
                        words[c + 1] |= pack_bits<OP_BOOL>(v + 32);
                    }
                }
            }
            if (!LEVEL) {
#pragma unroll
                for (int c = 0; c < CW; c++) out[0][c] = words[c];
            }
            }
            if (!ok) break;
            const int64_t row =
                (int64_t)tc.tm * LY::TILE_M + (int64_t)rank * BM + 32 * quarter + lane;
            if (LEVEL) {
                // quadrant (r, c) of the block's C: rows r m, words c n/64
                const int64_t w0 = (int64_t)tc.tn * (BN / 64) + chalf * (CW / 2);
                const int64_t nw = tc.n / 64;
                if (row < tc.m) {
#pragma unroll
                    for (int q = 0; q < (LEVEL ? 4 : 1); q++) {
                        uint64_t* crow = tc.C + ((q >> 1) * (int64_t)tc.m + row) * tc.ldc +
                                         (q & 1) * nw;
#pragma unroll
                        for (int c = 0; c < CW / 2; c++)
                            if (w0 + c < nw)
                                crow[w0 + c] = (uint64_t)qo[32 * (CW * q + 2 * c)] |
                                               ((uint64_t)qo[32 * (CW * q + 2 * c + 1)] << 32);
                    }
                }
            } else if (row < tc.m) {
                uint64_t* crow = tc.C + row * tc.ldc;
                const int64_t w0 = (int64_t)tc.tn * (BN / 64) + chalf * (CW / 2);
                const int64_t nw = tc.n / 64;
#pragma unroll
                for (int c = 0; c < CW / 2; c++)
                    if (w0 + c < nw)
                        crow[w0 + c] = (uint64_t)out[0][2 * c] | ((uint64_t)out[0][2 * c + 1] << 32);
            }
        }
        // a loop left early (a wait gave up) may still have an item copy in
        // flight into this warp's slot
        if (BATCHED) cp_async_wait_all();
    }

    tc_fence_before();
    __syncthreads();
    // A pair leaves together: the peer's remote arrivals and the MMAs that
    // read its shared memory and TMEM are over before either CTA frees TMEM.
    if (PAIR) cluster_sync();
    if (warp == MMA_WARP) {
        tc_fence_after();
        tmem_dealloc<PAIR>(tmem);
    }
}

// ---------------------------------------------------------------- host side
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)f;
    });
    return fn;
}

}  // namespace

// 3-D map over uint64 words: (k/64 words, rows, leaves), box (box_words,
// box_rows, 1). Boxes that run past k or the rows are zero-filled, which
// adds nothing to the counts.
bool tc_make_map(CUtensorMap* map, const uint64_t* base, int64_t kwords, int64_t rows,
                 int64_t pitch, int64_t count, int64_t stride, int box_rows, int box_words,
                 bool swizzle64) {
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {(cuuint64_t)kwords, (cuuint64_t)rows, (cuuint64_t)count};
    const int64_t leaf_stride = count > 1 ? stride : rows * pitch;
    cuuint64_t strides[2] = {(cuuint64_t)(pitch * 8), (cuuint64_t)(leaf_stride * 8)};
    cuuint32_t box[3] = {(cuuint32_t)box_words, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 3, (void*)base, dims, strides, box,
                          estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          swizzle64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

namespace {

constexpr int MAX_DEVICES = 64;

int current_device() {
    int d = 0;
    cudaGetDevice(&d);
    return d;
}

// Per-device one-time setup (function attributes and occupancy are per device).
std::mutex g_setup_mu;

template <bool BATCHED, bool PAIR, bool LEVEL = false>
cudaError_t set_smem_attr() {
    static bool done[MAX_DEVICES] = {false};
    static cudaError_t err[MAX_DEVICES];
    const int d = current_device();
    if (d < 0 || d >= MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_setup_mu);
    if (!done[d]) {
        err[d] = cudaFuncSetAttribute(tc_nt_kernel<BATCHED, PAIR, LEVEL>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      Lay<PAIR, LEVEL>::SMEM_BYTES);
        done[d] = true;
    }
    return err[d];
}

cudaLaunchConfig_t pair_config(unsigned units, size_t smem, cudaLaunchAttribute* at) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * units);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = smem;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

// CTA pairs of the e4m3 kernel (or, LEVEL, of the in-kernel-level kernel on
// e2m1 operands) that can be resident at once on the current device (clusters
// of two on one TPC); 0 if cluster launches are unavailable.
template <bool LEVEL>
int pair_slots() {
    static int slots[MAX_DEVICES];
    static bool done[MAX_DEVICES] = {false};
    const int d = current_device();
    if (d < 0 || d >= MAX_DEVICES) return 0;
    if (set_smem_attr<false, true, LEVEL>() != cudaSuccess) return 0;
    std::lock_guard<std::mutex> lk(g_setup_mu);
    if (!done[d]) {
        cudaLaunchAttribute at[1];
        const cudaLaunchConfig_t cfg =
            pair_config((unsigned)sm_count(), Lay<true, LEVEL>::SMEM_BYTES, at);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, tc_nt_kernel<false, true, LEVEL>, &cfg) !=
            cudaSuccess) {
            (void)cudaGetLastError();
            n = 0;
        }
        slots[d] = n;
        done[d] = true;
    }
    return slots[d];
}

// units: CTAs (single) or CTA pairs (PAIR) to launch.
template <bool BATCHED, bool PAIR, bool LEVEL = false>
cudaError_t launch_tc(const CUtensorMap& ma, const CUtensorMap& mb, const Params& prm, int units,
                      cudaStream_t s) {
    const cudaError_t e = set_smem_attr<BATCHED, PAIR, LEVEL>();
    if (e != cudaSuccess) return e;
    if (!PAIR) {
        tc_nt_kernel<BATCHED, false>
            <<<units, THREADS, Lay<false>::SMEM_BYTES, s>>>(ma, mb, prm);
        return cudaGetLastError();
    }
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = pair_config((unsigned)units, Lay<PAIR, LEVEL>::SMEM_BYTES, at);
    cfg.stream = s;
    return cudaLaunchKernelEx(&cfg, tc_nt_kernel<BATCHED, PAIR, LEVEL>, ma, mb, prm);
}

Spread spread_factors() {
    Spread sp;
    for (int j = 0; j < 8; j++) sp.f[j] = j <= 3 ? (1u << (3 - j)) : (1u << (35 - j));
    sp.g[0] = 2u;
    sp.g[1] = 1u;
    sp.g[2] = 1u << 31;
    sp.g[3] = 1u << 30;
    return sp;
}

}  // namespace

bool tc_path_available() { return device_cc() == 103 && encode_fn() != nullptr; }

// SM pairs need cluster launches with both CTAs of a pair resident at once.
bool tc_pair_available() { return tc_path_available() && pair_slots<false>() > 0; }
bool tc_fp4_available() { return tc_path_available() && tc_fp4_slots() > 0; }

// Longest run of k stages accumulated before the counts are flushed from
// TMEM: both formats read parity through an FP32 value count * 2^-12, exact
// while count < 2^23: at most 65534 stages of 128 k (e4m3), or 32766 of 256
// (e2m1, the in-kernel level). A multiple of the operand stages per packed
// stage (flushes happen between packed stages).
int tc_kchunk_stages(bool fp4, int nks) {
    const int cap = fp4 ? 32766 : 65534;
    return nks < cap ? nks : cap;
}

bmm_status run_tc_strided(int op, int path, const uint64_t* A, int64_t lda, int64_t strideA,
                          const uint64_t* Bt, int64_t ldb, int64_t strideB, uint64_t* C,
                          int64_t ldc, int64_t strideC, int64_t count, int64_t m, int64_t k,
                          int64_t n, cudaStream_t s) {
    const bool fp4 = path == BMM_PATH_TC_FP4_PAIR;
    const bool pair = fp4 || path == BMM_PATH_TC_FP8_PAIR;
    if (!tc_path_available() || (path != BMM_PATH_TC_FP8 && !pair)) return BMM_ERR_UNSUPPORTED;
    if (k % KS_MIN || (lda & 1) || (ldb & 1) ||
        (count > 1 && ((strideA & 1) || (strideB & 1))))
        return BMM_ERR_UNSUPPORTED;
    if (m <= 0 || n <= 0 || k <= 0 || count <= 0) return BMM_OK;
    // tile and stage indices are 32-bit in the kernel
    if (m > 0x7fffffffLL || n > 0x7fffffffLL || k / KS_MIN > 0x3fffffffLL)
        return BMM_ERR_UNSUPPORTED;
    if (fp4)
        return run_fp4_strided(op, A, lda, strideA, Bt, ldb, strideB, C, ldc, strideC, count, m, k,
                               n, s);
    const int slots = pair ? pair_slots<false>() : sm_count();
    if (slots <= 0) return BMM_ERR_UNSUPPORTED;
    uint32_t* err = device_error_word();
    if (!err) return BMM_ERR_NOMEM;
    const int64_t kp = SUB * KS_MIN;  // k bits per packed stage
    const int tile_m = pair ? Lay<true>::TILE_M : Lay<false>::TILE_M;
    const int brows = pair ? Lay<true>::BROWS : Lay<false>::BROWS;
    CUtensorMap ma, mb;
    if (!tc_make_map(&ma, A, k / 64, m, lda, count, strideA, BM, (int)(kp / 64)) ||
        !tc_make_map(&mb, Bt, k / 64, n, ldb, count, strideB, brows, (int)(kp / 64)))
        return BMM_ERR_CUDA;
    Params prm{};
    prm.C = C;
    prm.ldc = ldc;
    prm.strideC = strideC;
    prm.m = (int)m;
    prm.n = (int)n;
    prm.nks = (int)((k + kp - 1) / kp) * SUB;  // whole packed stages; the tail is zero-filled
    prm.op = op;
    prm.kchunk = tc_kchunk_stages(false, prm.nks);
    prm.tiles_m = (int)((m + tile_m - 1) / tile_m);
    prm.tiles_n = (int)((n + BN - 1) / BN);
    const int64_t total = (int64_t)prm.tiles_m * prm.tiles_n * count;
    if (total > 0x7fffffff) return BMM_ERR_UNSUPPORTED;
    prm.total_tiles = (int)total;
    prm.err = err;
    prm.sp = spread_factors();
    TraceScope ts(BMM_PHASE_BASE, s);
    const int units = prm.total_tiles < slots ? prm.total_tiles : slots;
    const cudaError_t e = pair ? launch_tc<false, true>(ma, mb, prm, units, s)
                               : launch_tc<false, false>(ma, mb, prm, units, s);
    if (e != cudaSuccess) return cuda_fail(e);
    return BMM_OK;
}

// The binary product of each block of a batch through one Strassen level run
// inside the e2m1 SM-pair kernel: block h is C (m x n, pitch ldc) = A (m x k,
// pitch lda) times Bt (n x k, pitch ldb)^T at A + h strideA, Bt + h strideB,
// C + h strideC (words). m and n even, k a multiple of 2 x 512 bits (every
// quadrant's k whole packed stages, so no copy reads into the neighbouring
// quadrant), even pitches and strides.
bmm_status run_tc_level(const uint64_t* A, int64_t lda, int64_t strideA, const uint64_t* Bt,
                        int64_t ldb, int64_t strideB, uint64_t* C, int64_t ldc, int64_t strideC,
                        int64_t count, int64_t m, int64_t k, int64_t n, const LevelMasks& masks,
                        cudaStream_t s) {
    using LY = Lay<true, true>;
    if (!tc_path_available()) return BMM_ERR_UNSUPPORTED;
    if (m % 2 || n % 2 || k % (2 * LY::KP) || (lda & 1) || (ldb & 1) ||
        (count > 1 && ((strideA & 1) || (strideB & 1))))
        return BMM_ERR_UNSUPPORTED;
    if (m <= 0 || n <= 0 || k <= 0 || count <= 0) return BMM_OK;
    if (m > 0x7fffffffLL || n > 0x7fffffffLL || k / KS_MIN > 0x3fffffffLL)
        return BMM_ERR_UNSUPPORTED;
    const int slots = pair_slots<true>();
    if (slots <= 0) return BMM_ERR_UNSUPPORTED;
    uint32_t* err = device_error_word();
    if (!err) return BMM_ERR_NOMEM;
    const int64_t hm = m / 2, hk = k / 2, hn = n / 2;
    CUtensorMap ma, mb;
    if (!tc_make_map(&ma, A, k / 64, m, lda, count, strideA, BM, LY::KP / 64) ||
        !tc_make_map(&mb, Bt, k / 64, n, ldb, count, strideB, LY::BROWS, LY::KP / 64))
        return BMM_ERR_CUDA;
    Params prm{};
    prm.C = C;
    prm.ldc = ldc;
    prm.strideC = strideC;
    prm.m = (int)hm;
    prm.n = (int)hn;
    prm.nks = (int)(hk / LY::KP) * SUB;
    prm.op = OP_GF2;
    prm.kchunk = tc_kchunk_stages(true, prm.nks);
    prm.tiles_m = (int)((hm + LY::TILE_M - 1) / LY::TILE_M);
    prm.tiles_n = (int)((hn + BN - 1) / BN);
    const int64_t total = (int64_t)prm.tiles_m * prm.tiles_n * count;
    if (total > 0x7fffffff / 7) return BMM_ERR_UNSUPPORTED;
    prm.total_tiles = (int)total;
    prm.err = err;
    prm.sp = spread_factors();
    for (int h = 0; h < 7; h++) {
        // a packed stage holds at most QTILES quadrant tiles (every variant's
        // products combine at most six)
        if (__builtin_popcount(masks.xi[h] & 0xFu) + __builtin_popcount(masks.eta[h] & 0xFu) >
            LY::QTILES)
            return BMM_ERR_UNSUPPORTED;
        prm.xi4 |= (masks.xi[h] & 0xFu) << (4 * h);
        prm.eta4 |= (masks.eta[h] & 0xFu) << (4 * h);
    }
    for (int q = 0; q < 4; q++) prm.zeta7 |= (masks.zeta[q] & 0x7Fu) << (7 * q);
    prm.qkw = (int)(hk / 64);
    TraceScope ts(BMM_PHASE_BASE, s);
    const int units = prm.total_tiles < slots ? prm.total_tiles : slots;
    const cudaError_t e = launch_tc<false, true, true>(ma, mb, prm, units, s);
    if (e != cudaSuccess) return cuda_fail(e);
    return BMM_OK;
}

}  // namespace bmm

namespace bmm {

int tc_pair_slots(bool fp4) {
    if (!tc_path_available()) return 0;
    return fp4 ? tc_fp4_slots() : pair_slots<false>();
}

bool tc_make_problem(TcProblem* out, const uint64_t* A, int64_t lda, const uint64_t* Bt,
                     int64_t ldb, uint64_t* C, int64_t ldc, int64_t m, int64_t k, int64_t n,
                     int op, bool pair, bool fp4) {
    if (k % KS_MIN || (lda & 1) || (ldb & 1) || (fp4 && !pair)) return false;
    const int64_t kp = SUB * KS_MIN;
    if (fp4 ? !tc_fp4_maps(&out->mapA, &out->mapB, A, lda, 0, Bt, ldb, 0, 1, m, k, n)
            : !tc_make_map(&out->mapA, A, k / 64, m, lda, 1, 0, BM, (int)(kp / 64)) ||
                  !tc_make_map(&out->mapB, Bt, k / 64, n, ldb, 1, 0,
                               pair ? Lay<true>::BROWS : Lay<false>::BROWS,
                               (int)(kp / 64)))
        return false;
    out->C = C;
    out->ldc = ldc;
    out->m = (int32_t)m;
    out->n = (int32_t)n;
    out->nks = fp4 ? (int32_t)((k + 127) / 128) : (int32_t)(((k + kp - 1) / kp) * SUB);
    out->op = op;
    return true;
}

cudaError_t tc_prepare_batched(bool pair, bool fp4) {
    if (fp4 && !pair) return cudaErrorInvalidValue;
    return fp4    ? tc_fp4_prepare_batched()
           : pair ? set_smem_attr<true, true>()
                  : set_smem_attr<true, false>();
}

cudaError_t tc_launch_batched(const TcProblem* d_probs, const TcWorkItem* d_items,
                              const int32_t* d_unit_ptr, int units, bool pair, bool fp4,
                              cudaStream_t s) {
    if (fp4) return pair ? tc_fp4_launch_batched(d_probs, d_items, d_unit_ptr, units, s)
                         : cudaErrorInvalidValue;
    uint32_t* err = device_error_word();
    if (!err) return cudaErrorMemoryAllocation;
    Params prm{};
    prm.probs = d_probs;
    prm.items = d_items;
    prm.cta_ptr = d_unit_ptr;
    prm.kchunk = tc_kchunk_stages(false, 0x7fffffff);
    prm.err = err;
    prm.sp = spread_factors();
    CUtensorMap dummy;
    std::memset(&dummy, 0, sizeof(dummy));
    TraceScope ts(BMM_PHASE_BASE, s);
    return pair ? launch_tc<true, true>(dummy, dummy, prm, units, s)
                : launch_tc<true, false>(dummy, dummy, prm, units, s);
}

}  // namespace bmm

extern "C" bmm_status bmm_selftest_wait_timeout(int64_t limit_ns, bmm_stream_t stream) {
    using namespace bmm;
    if (limit_ns <= 0 || limit_ns > 10000000000LL) return BMM_ERR_INVALID;
    uint32_t* err = device_error_word();
    if (!err) return BMM_ERR_NOMEM;
    wait_selftest_kernel<<<1, 1, 0, (cudaStream_t)stream>>>(err, (uint64_t)limit_ns);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? BMM_OK : cuda_fail(e);
}
