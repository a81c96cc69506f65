// Tensor-core base case on e2m1 operands (BMM_PATH_TC_FP4_PAIR) for sm_103a:
// C = A * Bt^T over GF(2) or the Boolean algebra (Sec. 3.10 inner layer), A
// (m x k) and Bt (n x k) packed along k.
//
// The bit product is an integer dot product of 0/1 vectors: GF(2) takes it
// mod 2, Boolean takes it > 0. Every bit becomes a 4-bit e2m1 value and the
// tensor cores count exactly with kind::mxf4 MMAs of K = 96, the dense K that
// sm_103a alone has: 128 cycles for M = 256, N = 256 on an SM pair, the same
// as K = 64 takes (measured: 24545 against 16364 MACs per clock per SM).
//
// Two CTAs of a cluster on two SMs share one 256 x 256 tile of C
// (cta_group::2). Each expands its own 128 rows of A into its TMEM and its
// own half of the tile's Bt rows into its shared memory; the even CTA issues
// the MMAs, which read both CTAs' operands and accumulate each CTA's 128 rows
// in its own TMEM. Persistent, one CTA per SM, 28 warps:
//   warp 0       MMA issuer (the even CTA's).
//   warp 1       TMA producer: packed tiles of A and Bt, PSTAGES deep. A stage
//                is 384 bits of k, four MMAs, in rows of 64 bytes.
//   warps 4-11   Bt expansion, two groups of four; the groups take the stages
//                in turn, so the latencies of one stage (two barriers, the
//                shared loads, the proxy fence) overlap the other group's work.
//   warps 12-19  A expansion, two groups likewise, one warp per TMEM lane
//                quarter.
//   warps 20-27  epilogue: accumulator -> parity or non-zero bits -> 64-bit words.
// Expanded stages go to four operand slots (A in TMEM, Bt in shared memory).
//
// What bounds it: large products the MMA pipe at the clock that the power limit
// leaves (1.8 to 1.95 GHz; with the A loads, half of Bt's stores or the proxy
// fence left out 8192^3 loses less than 1 %); short k the hand-off of the one
// accumulator at the end of a tile and the epilogue; one tile alone the
// expansion's loop (525 cycles a stage against the MMAs' 512). The roles share
// the SM's instruction issue, hence the short loops that are not unrolled over
// stages, an issuer that reads the next slot's barrier while it issues, and an
// expansion that loads the group's next stage while it stores this one.
//
// Measured, us inside a graph, transpose of B included, GF(2) / Boolean:
// 16384 x k x 16384 at k = 256 52.6 / 56.4, 1024 73.6 / 76.7, 4096 192 / 195, 8192
// 358, 32768 1314 (1.34e16 operations a second; 2310 with K = 64 MMAs); 8192^3 96,
// 4096^3 20.3, 2048^3 8.9, 16384 x 12288 x 192 15.9, 64 x 2048 x 32768 14.6,
// 256 x 512 x 384 6.8.
//
// The TMA side would be a bound of its own with 48-byte box rows and copies
// issued from one lane of a divergent warp (ROW_BYTES and the producer below):
// 64 x 2048 x 32768 took 26.5 us so, 16384 x 12288 x 192 18.5. Other forms of the
// expansion were slower too: two slots per issue block, issue from one lane of
// a divergent warp (1.8 times at k = 32768), shifts as multiplications on the
// FMA pipe (1.04 times).
//
// The hand-off: the MMAs of the next tile wait until the epilogue has read the
// accumulator (the operand slots and the scales leave no TMEM for a second
// one); every 100 cycles of it are 3 % at k = 1024. So every count carries a start
// value that puts it into the low half of its word, two packed loads bring a
// warp's 128 columns at once, and the accumulator goes back before anything is
// packed (packing 32 columns at a time first took 920 cycles, Boolean 1700, of a
// 4096-bit tile's 7460). The epilogue then has one 16-byte store a lane (stores
// of 8 bytes, each to 32 rows, were what bounded k = 1024: they share a pipe with
// the expansion's shared memory traffic) and multiplications for the divisions
// in a tile's place; one block of issue code serves all stages, the last of a
// tile too.
//
// The hand-off was not shortened by: an accumulator in two halves of 128 columns,
// one drained while the other's MMAs run (N = 128 MMAs are as fast as N = 256 ones,
// but the issuing warp's longer code ran from a cold instruction cache, some 80
// cycles an MMA: 1.2 times the time at k = 1024); two loads of 64 columns instead of
// 128 at once, for registers (1.13 times); a relaxed arrive on the accumulator's
// barrier, an issuer that spins on its barriers, the expansion in functions of
// its own (no change); setmaxnreg (ptxas finds no allocation).
//
// Within every 128-bit vector of k the expansion permutes k, the same way in
// A and Bt, so the contraction is unchanged. Every mbarrier wait is bounded
// (about 2 s); a wait that gives up records DEVERR_TIMEOUT and makes its role
// stop; the CTA then drains its own copies and MMAs (bounded too), frees TMEM
// and returns.
#include <cuda.h>

#include <cstring>
#include <mutex>

#include "pdl.cuh"
#include "plan.h"
#include "tc_batched.h"
#include "tc_ptx.cuh"

namespace bmm {
namespace {

constexpr int BM = TC_TILE_M;          // rows of C per CTA (its TMEM lanes)
constexpr int TILE_M = 2 * BM;         // rows of C per pair
constexpr int BROWS = BN / 2;          // Bt rows per CTA
// 128-bit vectors of k per stage (384 bits: four MMAs).
constexpr int STAGE_VECS = 3;
// A packed row of a stage is a window of 64 bytes that starts 32-byte aligned
// in its row of k, so every other stage's three vectors begin one vector into
// it. The TMA unit takes about a cycle for a box row that is aligned to its 64
// bytes, 1.25 where it starts at the half, but 3 where it starts at an odd
// multiple of 16 bytes (48- and 64-byte rows alike, measured): with boxes of
// the 48 bytes alone a stage's 256 rows took 514 cycles, as long as its MMAs.
// The 64-byte swizzle puts the 16-byte loads of eight adjacent rows on eight
// different bank groups.
constexpr int ROW_BYTES = 64;
constexpr int SLOTS = 4;               // operand slots (expanded stages)
constexpr int MMA_COLS = 12;           // TMEM columns of A per MMA (96 nibbles a row)
constexpr int SLOT_COLS = 4 * MMA_COLS;
constexpr int A_COL = BN;              // accumulator in columns [0, BN), then the A slots
// Block scales of A and of Bt, eight columns each (uniform, so their layout
// over rows and blocks does not matter), then those of the bias MMA and its A
// operand.
constexpr int SF_COL = 448, SF_COLS = 8;
constexpr int BIAS_SF_COL = SF_COL + 2 * SF_COLS;
constexpr int ONE_SF_COL = BIAS_SF_COL + 2 * SF_COLS;  // A's scales where every element is 1.0
constexpr int BIAS_A_COL = ONE_SF_COL + SF_COLS;
static_assert(A_COL + SLOTS * SLOT_COLS <= SF_COL && BIAS_A_COL + MMA_COLS <= TMEM_COLS,
              "TMEM budget");
// Bt in shared memory: unswizzled K-major core matrices (8 rows x 16 bytes),
// row groups 128 bytes apart, the 16-byte chunks along k CHUNK_BYTES apart. A
// lane per row then writes 16-byte chunks of adjacent rows side by side.
constexpr int CHUNK_BYTES = BROWS * 16;
constexpr int EB_BYTES = 4 * STAGE_VECS * CHUNK_BYTES;
constexpr int PSTAGES = 6;             // packed stages; even, so that each is one group's
constexpr int PA_BYTES = BM * ROW_BYTES;
constexpr int PB_BYTES = BROWS * ROW_BYTES;
constexpr int GROUP_WARPS = 4;
constexpr int MMA_WARP = 0, TMA_WARP = 1, BEXP_WARP0 = 4, AEXP_WARP0 = 12, EPI_WARP0 = 20;
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 28 * 32;
constexpr int NBARS = 2 * PSTAGES + 2 * SLOTS + 3;
constexpr int ITEM_BYTES = 48;
constexpr int OFF_EB = 0;
constexpr int OFF_PA = OFF_EB + SLOTS * EB_BYTES;
constexpr int OFF_PB = OFF_PA + PSTAGES * PA_BYTES;
constexpr int OFF_BIAS = OFF_PB + PSTAGES * PB_BYTES;  // Bt operand of the bias MMA
constexpr int OFF_SKIP = OFF_BIAS + 3 * CHUNK_BYTES;   // per packed stage: bytes before its vectors
constexpr int OFF_ITEMS = OFF_SKIP + 32;
constexpr int OFF_BAR = OFF_ITEMS + EPI_WARPS * 2 * ITEM_BYTES;
constexpr int OFF_TMEM_SLOT = OFF_BAR + NBARS * 8;
constexpr int SMEM_BYTES = OFF_TMEM_SLOT + 16;
static_assert(PA_BYTES == PB_BYTES, "one stage stride for both operands");
static_assert(OFF_PA % 512 == 0 && PA_BYTES % 512 == 0 && 4 * PSTAGES <= 32, "swizzle atoms, skips");
static_assert(SMEM_BYTES <= 227 * 1024, "shared memory budget");
static_assert(sizeof(TcWorkItem) == ITEM_BYTES, "three 16-byte copies per item");
// Every accumulator starts at 2^11 and a count c adds c * 2^-12, so the FP32
// word is 0x45000000 + c while c < 2^23: its low 16 bits, which the packed
// TMEM loads bring two columns to a register, are c mod 2^16. The start value
// comes from one MMA per segment with a single non-zero element in every row
// of A and of Bt (1.0) and block scales of its own.
// Stages accumulated before the counts leave TMEM: parity needs c < 2^23, the
// non-zero test c < 2^16.
constexpr int KCHUNK_GF2 = ((1 << 23) - 1) / (128 * STAGE_VECS);
constexpr int KCHUNK_BOOL = ((1 << 16) - 1) / (128 * STAGE_VECS);

// UE8M0 block scales: 2^-6 (products of 1.0 count as 2^-12), and A's 2^-4, 2^-6
// and 2^-8 for the three kinds of block; 2^5 and 2^6.
constexpr uint32_t SCALES = 0x79797979u, SCALES_A = 0x7977797Bu;
constexpr uint32_t BIAS_SCALES_A = 0x84848484u, BIAS_SCALES_B = 0x85858585u;

// A whole warp's bounded wait for the phase of `bar` with the given parity:
// every lane gets the same answer, so a wait that gives up cannot leave a
// part of the warp behind at a later warp-wide instruction.
__device__ __noinline__ bool warp_wait_slow(uint32_t bar, uint32_t parity, uint32_t* err) {
    const uint64_t t0 = globaltimer();
    for (uint32_t i = 1;; i++) {
        if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
        if ((i & 255u) == 0 && __any_sync(0xffffffffu, globaltimer() - t0 > WAIT_NS)) {
            atomicOr(err, DEVERR_TIMEOUT);
            return false;
        }
    }
}
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, uint32_t* err) {
    if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
    return warp_wait_slow(bar, parity, err);
}

__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(p));
    return p != 0;
}

// Descriptor of a K-major operand in unswizzled core matrices.
__device__ __forceinline__ uint64_t smem_desc_plain(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(CHUNK_BYTES >> 4) << 16;  // LBO: the next 16 bytes of k
    d |= (uint64_t)(128 >> 4) << 32;          // SBO: the next 8 rows
    d |= (uint64_t)1 << 46;                   // descriptor version for tcgen05
    return d;
}

// Instruction descriptor: instr_desc_mxf4 with bit 31 (K = 96).
template <int N>
__host__ __device__ constexpr uint32_t instr_desc_k96() {
    return instr_desc_mxf4<TILE_M, N>() | (1u << 31);
}

// D (TMEM columns 0..) += A (TMEM columns a_col..) x B (shared, descriptor);
// BIAS: D = the start value of every count. The whole TMEM is allocated, so
// its columns count from 0. ONES: every element is 1.0.
enum { KINDS, ONES, BIAS };
template <int KIND>
__device__ __forceinline__ void mma_k96(uint32_t a_col, uint64_t db, uint32_t idesc) {
    constexpr uint32_t sfa = KIND == BIAS ? BIAS_SF_COL : KIND == ONES ? ONE_SF_COL : SF_COL;
    constexpr uint32_t sfb = (KIND == BIAS ? BIAS_SF_COL : SF_COL) + SF_COLS;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::mxf4.block_scale.block32"
        " [%6], [%0], %1, %2, [%3], [%4], p;\n\t}" ::"r"(a_col),
        "l"(db), "r"(idesc), "r"(sfa), "r"(sfb), "n"(KIND == BIAS ? 0 : 1), "r"(0)
        : "memory");
}

// The low halves of 128 columns (one row per thread): column 2 j of a register
// pair's 64 in the low, column 2 j + 1 in the high half of v[j]. Then wait for
// the loads.
__device__ __forceinline__ void tmem_ld128_low(uint32_t taddr, uint32_t (&v)[64]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.pack::16b.b32 {"
        "%0, %1, %2, %3, %4, %5, %6, %7, "
        "%8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, "
        "%24, %25, %26, %27, %28, %29, %30, %31}, [%64];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x32.pack::16b.b32 {"
        "%32, %33, %34, %35, %36, %37, %38, %39, "
        "%40, %41, %42, %43, %44, %45, %46, %47, "
        "%48, %49, %50, %51, %52, %53, %54, %55, "
        "%56, %57, %58, %59, %60, %61, %62, %63}, [%65];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
          "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]),
          "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]),
          "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]),
          "=r"(v[30]), "=r"(v[31]), "=r"(v[32]), "=r"(v[33]), "=r"(v[34]), "=r"(v[35]),
          "=r"(v[36]), "=r"(v[37]), "=r"(v[38]), "=r"(v[39]), "=r"(v[40]), "=r"(v[41]),
          "=r"(v[42]), "=r"(v[43]), "=r"(v[44]), "=r"(v[45]), "=r"(v[46]), "=r"(v[47]),
          "=r"(v[48]), "=r"(v[49]), "=r"(v[50]), "=r"(v[51]), "=r"(v[52]), "=r"(v[53]),
          "=r"(v[54]), "=r"(v[55]), "=r"(v[56]), "=r"(v[57]), "=r"(v[58]), "=r"(v[59]),
          "=r"(v[60]), "=r"(v[61]), "=r"(v[62]), "=r"(v[63])
        : "r"(taddr), "r"(taddr + 64)
        : "memory");
}

// 32 columns' result bits from their 16 packed registers. The deciding bit of a
// count is its lowest (for Boolean, that of min(count, 1)): a byte permute brings
// the low bytes of four columns into one register, and seven merges interleave
// eight of those, so that bit 8 b + i of the result is column 4 i + b. 22
// operations a word (and 16 minima for Boolean) against 32 (48) with a mask and a
// shifted add per register.
template <int OP>
__device__ __forceinline__ uint32_t pack_low(const uint32_t* v) {
    uint32_t t[8];
#pragma unroll
    for (int i = 0; i < 8; i++)
        t[i] = OP == OP_GF2 ? __byte_perm(v[2 * i], v[2 * i + 1], 0x6420)
                            : __byte_perm(__vminu2(v[2 * i], 0x00010001u),
                                          __vminu2(v[2 * i + 1], 0x00010001u), 0x6420);
#pragma unroll
    for (int j = 1; j < 8; j *= 2) {
        const uint32_t low = j == 1 ? 0x55555555u : j == 2 ? 0x33333333u : 0x0F0F0F0Fu;
#pragma unroll
        for (int i = 0; i < 8; i += 2 * j) t[i] = (t[i] & low) | ((t[i + j] << j) & ~low);
    }
    return t[0];
}
// The accumulator column (of each 32) that Bt row r (of each 32) must take for
// that.
__device__ __forceinline__ int column_of_row(int r) { return 4 * (r & 7) + (r >> 3); }

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
        "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]),
        "r"(v[15])
        : "memory");
}

// Packed word x holds 32 consecutive k of one row; word j of its expansion gets
// bits 4t + j of x in nibble t. Bits 0, 1 and 2 stay in their place and are the
// e2m1 values 0.5, 1.0 and 2.0; bit 3 (the sign place) moves to 1.0. A's and
// Bt's words come out alike: the products 0.25, 1 and 4 of two set bits are made
// one by the block scales, as each kind fills a block of 32.
__device__ __forceinline__ uint32_t spread(uint32_t x, int j) {
    return j < 3 ? x & (0x11111111u << j) : (x >> 2) & 0x22222222u;
}
__device__ __forceinline__ void spread4(const uint4& x, int j, uint32_t* y) {
    y[0] = spread(x.x, j);
    y[1] = spread(x.y, j);
    y[2] = spread(x.z, j);
    y[3] = spread(x.w, j);
}

__device__ __forceinline__ void red_xor(uint64_t* p, uint64_t v) {
    asm volatile("red.global.xor.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void red_or(uint64_t* p, uint64_t v) {
    asm volatile("red.global.or.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
        : "memory");
}

// The kernel's forms: one shape, `count` leaves side by side; one shape with
// slices of k; products of any shapes.
enum { WHOLE, SLICED, BATCHED };

struct Params {
    // WHOLE and SLICED: one shape, `count` leaves side by side
    uint64_t* C;
    int64_t ldc;
    // Words between leaves; SLICED (which has one leaf), as the batched form's code
    // suffers from longer parameters: the vectors of a slice, and above 2^32
    // 2^16 / sliced tiles, rounded up.
    int64_t strideC;
    int whole;  // SLICED: tiles before the sliced ones
    int m, n, nvec, op;  // nvec: 128-bit vectors of k
    TileOrder order;
    int items_total;       // tiles and slices
    // BATCHED: per-problem descriptors and per-pair work lists
    const TcProblem* probs;
    const TcWorkItem* items;
    const int32_t* unit_ptr;
    uint32_t* err;
};

// Everything a role needs about one output tile.
struct Tile {
    const CUtensorMap* ma;
    const CUtensorMap* mb;
    uint64_t* C;
    int64_t ldc;
    int m, n, nvec, op, tm, tn, leaf;  // leaf: SLICED: first vector of k

    int n128;  // the tile's columns past 128 lie beyond n: N = 128 MMAs
};

__device__ __forceinline__ int unit_id() { return (int)(blockIdx.x >> 1); }
__device__ __forceinline__ int unit_count() { return (int)(gridDim.x >> 1); }

__device__ __forceinline__ Tile item_tile(const Params& p, const TcWorkItem& w) {
    const TcProblem* d = p.probs + w.prob;
    return {&d->mapA, &d->mapB, w.C, w.ldc, w.m, w.n, w.nks, w.op, w.tm, w.tn, 0, w.n128};
}

// One shape: the unit's idx-th item, nvec vectors of k of a tile from v0 on. SLICED:
// whole tiles, then (at most one a unit) slices of the tiles after them, slice by
// slice.
struct Item {
    TileCoord c;
    int v0, nvec;
};
template <int FORM>
__device__ __forceinline__ Item get_item(const Params& p, int idx) {
    const int i = unit_id() + idx * unit_count();
    if (FORM != SLICED) return {p.order.tile(i), 0, p.nvec};
    const int tiles = (int)p.order.per_leaf.d;
    int tile = i, v0 = 0, nvec = p.nvec;
    if (i >= p.whole) {
        // ((i - whole) / sliced tiles: both are below 2^8)
        const int slice = (int)((uint32_t)(i - p.whole) * (uint32_t)(p.strideC >> 32) >> 16);
        tile = i - slice * (tiles - p.whole);
        v0 = slice * (int)(uint32_t)p.strideC;
        nvec = min(p.nvec - v0, (int)(uint32_t)p.strideC);
    }
    return {p.order.tile(tile), v0, nvec};
}

template <int FORM>
__device__ __forceinline__ Tile get_tile(const Params& p, const TcWorkItem* items, int idx,
                                         const CUtensorMap* ma, const CUtensorMap* mb) {
    if (FORM == BATCHED) return item_tile(p, items[idx]);
    const Item it = get_item<FORM>(p, idx);
    return {ma,
            mb,
            FORM == SLICED ? p.C : p.C + (int64_t)it.c.leaf * p.strideC,
            p.ldc,
            p.m,
            p.n,
            it.nvec,
            p.op,
            it.c.tm,
            it.c.tn,
            FORM == SLICED ? it.v0 : it.c.leaf,
            p.n - it.c.tn * BN <= BN / 2};
}

// Stages between flushes of the accumulator.
__device__ __forceinline__ int chunk_of(int op) {
    return op == OP_GF2 ? KCHUNK_GF2 : KCHUNK_BOOL;
}

// What the MMA issuer needs of a tile.
struct TileK {
    int nvec, n128, chunk;
};
template <int FORM>
__device__ __forceinline__ TileK get_tile_k(const Params& p, const TcWorkItem* items, int idx) {
    if (FORM == BATCHED) return {items[idx].nks, items[idx].n128, chunk_of(items[idx].op)};
    const bool narrow = (p.n - 1) % BN < BN / 2;  // some column tile is
    if (FORM == WHOLE && !narrow) return {p.nvec, 0, chunk_of(p.op)};
    const Item it = get_item<FORM>(p, idx);
    return {it.nvec, narrow && p.n - it.c.tn * BN <= BN / 2, chunk_of(p.op)};
}

template <int FORM>
__global__ void __launch_bounds__(THREADS, 1)
    tc_fp4_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  const Params p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = sbase + OFF_BAR;
    auto full_p = [&](int s) { return bar0 + 8u * s; };
    auto empty_p = [&](int s) { return bar0 + 8u * (PSTAGES + s); };
    auto full_o = [&](uint32_t q) { return bar0 + 8u * (2 * PSTAGES + q); };
    auto empty_o = [&](uint32_t q) { return bar0 + 8u * (2 * PSTAGES + SLOTS + q); };
    const uint32_t acc_full = bar0 + 8u * (2 * PSTAGES + 2 * SLOTS);
    const uint32_t acc_empty = acc_full + 8u;
    const uint32_t drain_bar = acc_full + 16u;

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    // CTA 0 issues the MMAs and holds the barriers that gate them (full_o,
    // acc_empty); both CTAs' producers and epilogues arrive there.
    const uint32_t rank = cluster_rank();

    if (threadIdx.x == 0) {
        for (int s = 0; s < PSTAGES; s++) {
            mbar_init(full_p(s), 1);
            mbar_init(empty_p(s), 2 * GROUP_WARPS);  // one group of each expansion
        }
        for (int q = 0; q < SLOTS; q++) {
            mbar_init(full_o(q), 2 * 2 * GROUP_WARPS);  // both CTAs
            mbar_init(empty_o(q), 1);
        }
        mbar_init(acc_full, 1);
        mbar_init(acc_empty, 2 * EPI_WARPS);
        mbar_init(drain_bar, 1);
        fence_barrier_init();
    }
    if (warp == MMA_WARP) tmem_alloc<true>(sbase + OFF_TMEM_SLOT);
    if (FORM != BATCHED && warp == TMA_WARP && lane == 0) {
        prefetch_tensormap(&tmA);
        prefetch_tensormap(&tmB);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // the peer's barriers exist before anything arrives on them
    tc_fence_after();

    int my_tiles = 0;
    const TcWorkItem* my_items = nullptr;
    int stages = 0;  // stages of k this pair runs
    if (FORM == BATCHED) {
        my_items = p.items + p.unit_ptr[unit_id()];
        my_tiles = p.unit_ptr[unit_id() + 1] - p.unit_ptr[unit_id()];
        stages = p.unit_ptr[unit_count() + 1 + unit_id()];
    } else {
        my_tiles = (p.items_total - unit_id() + unit_count() - 1) / unit_count();
        stages = my_tiles * ((p.nvec + STAGE_VECS - 1) / STAGE_VECS);
        if (FORM == SLICED && my_tiles > 0)  // (only the last item can be a slice)
            stages += (get_item<FORM>(p, my_tiles - 1).nvec + STAGE_VECS - 1) / STAGE_VECS -
                      (p.nvec + STAGE_VECS - 1) / STAGE_VECS;
    }

    // Every role waits for the pass that writes the operands, so that no bounded
    // wait runs while that pass does.
    if (warp >= BEXP_WARP0 && warp < EPI_WARP0) {
        // ------------------------------------------------ operand expansion
        const bool is_b = warp < AEXP_WARP0;
        const int group = (warp >> 2) & 1, quarter = warp & 3;
        // The row each lane expands. Bt rows go to the accumulator columns that
        // the epilogue's packing wants, so its lanes take them in an order that
        // keeps both the packed loads (swizzled rows of 64 bytes) and the 16-byte
        // stores of every eight lanes on different banks.
        const int blk = (lane >> 1) & 3;
        const int brow = 8 * blk + 2 * (((lane >> 3) + blk) & 3) + (lane & 1);
        const int row = 32 * quarter + (is_b ? brow : lane);
        const int bcol = 32 * quarter + column_of_row(brow);
        const uint32_t tlane = (uint32_t)(32 * quarter) << 16;
        if (group == 0) {
            // block scales and the bias operands, before the first full_o arrive
            if (is_b) {
                uint8_t* bias = smem + OFF_BIAS + (32 * quarter + lane) * 16;
#pragma unroll
                for (int c = 0; c < 3; c++)
                    *reinterpret_cast<uint4*>(bias + c * CHUNK_BYTES) =
                        make_uint4(c == 0 ? 2u : 0u, 0u, 0u, 0u);
                fence_proxy_async();
            } else {
                uint32_t f[16];
#pragma unroll
                for (int i = 0; i < 16; i++) f[i] = i < 8 ? SCALES_A : SCALES;
                tmem_st16(tlane + (uint32_t)SF_COL, f);
#pragma unroll
                for (int i = 0; i < 16; i++) f[i] = i < 8 ? BIAS_SCALES_A : BIAS_SCALES_B;
                tmem_st16(tlane + (uint32_t)BIAS_SF_COL, f);
#pragma unroll
                for (int i = 0; i < 16; i++) f[i] = i == 0 ? 2u : 0u;
                tmem_st16(tlane + (uint32_t)BIAS_A_COL, f);
#pragma unroll
                for (int i = 0; i < 16; i++) f[i] = SCALES;
                tmem_st8(tlane + (uint32_t)ONE_SF_COL, f);
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            }
        }
        // the packed row's first vector, the swizzle applied (its bits 4 and 5)
        const uint32_t src = (uint32_t)(row * ROW_BYTES + (row >> 1 & 3) * 16);
        const uint8_t* packed = smem + (is_b ? OFF_PB : OFF_PA);
        wait_for_operands();
        int s = group;           // packed stage
        uint32_t s_parity = 0;
        uint4 x[STAGE_VECS];
        auto load = [&](int at) {
            const uint32_t skip = *reinterpret_cast<const uint32_t*>(smem + OFF_SKIP + 4 * at);
#pragma unroll
            for (int v = 0; v < STAGE_VECS; v++)
                x[v] = *reinterpret_cast<const uint4*>(packed + at * PA_BYTES + (src ^ (skip + 16 * v)));
        };
        // whether x holds this stage's words already, and its slot has been seen free
        bool loaded = false, slot_free = false;
#pragma unroll 1
        for (int st = group; st < stages; st += 2) {
            const int q = st & (SLOTS - 1);
            if (!loaded) {
                if (!warp_wait(full_p(s), s_parity, p.err)) break;
                load(s);
            }
            if (!slot_free && !warp_wait(empty_o(q), ((st / SLOTS) & 1) ^ 1, p.err)) break;
            if (is_b) {
                uint8_t* eb = smem + OFF_EB + q * EB_BYTES + bcol * 16;
                // MMA v: the three unmoved kinds of vector v; MMA 3: the moved ones
#pragma unroll
                for (int v = 0; v < STAGE_VECS; v++)
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        uint32_t y[4];
                        spread4(x[v], j, y);
                        *reinterpret_cast<uint4*>(eb + (j < 3 ? 3 * v + j : 9 + v) * CHUNK_BYTES) =
                            make_uint4(y[0], y[1], y[2], y[3]);
                    }
            } else {
                tc_fence_after();  // the slot's MMAs, before our TMEM stores
#pragma unroll
                for (int c = 0; c < 12; c += 4) {  // 16 columns at a time
                    uint32_t y[16];
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        const int at = c + i, v = at < 9 ? at / 3 : at - 9, j = at < 9 ? at % 3 : 3;
                        spread4(x[v], j, y + 4 * i);
                    }
                    tmem_st16(tlane + (uint32_t)(A_COL + q * SLOT_COLS + 4 * c), y);
                }
            }
            // The packed stage goes back once its words have been used: an arrive
            // right behind the loads can overtake them, and the next TMA copy
            // then overwrites rows that have not been read (measured: about one
            // product in 2048 had a few wrong words).
            const int done = s;
            s += 2;
            if (s >= PSTAGES) {
                s -= PSTAGES;
                s_parity ^= 1;
            }
            // the group's next stage, where it is there: its loads overlap the
            // stores above
            const bool more = st + 2 < stages;
            const uint32_t next_full = mbar_test(full_p(s), s_parity);
            const uint32_t next_free = mbar_test(empty_o((st + 2) & (SLOTS - 1)), (((st + 2) / SLOTS) & 1) ^ 1);
            loaded = more && __all_sync(0xffffffffu, next_full);
            slot_free = __all_sync(0xffffffffu, next_free);
            if (loaded) load(s);
            if (is_b) {
                fence_proxy_async();
            } else {
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
            }
            __syncwarp();
            if (lane == 0) {
                mbar_arrive_cluster(full_o(q), 0);
                mbar_arrive(empty_p(done));
            }
        }
    } else if (warp >= EPI_WARP0) {
        // ---------------------------------------------------- epilogue
        // Two warps per TMEM lane quarter, each 128 columns.
        const int quarter = warp & 3;
        const int chalf = (warp - EPI_WARP0) >> 2;
        const uint32_t tlane = (uint32_t)(32 * quarter) << 16;
        constexpr int CW = 4;  // 32-column words per warp
        int seg = 0;
        bool ok = true;
        // batched: each tile's work item is copied into this warp's shared
        // slot while the tile before it runs
        const uint32_t islot =
            sbase + (uint32_t)(OFF_ITEMS + (warp - EPI_WARP0) * 2 * ITEM_BYTES);
        auto fetch_item = [&](int idx) {
            if (lane < 3)
                cp_async16(islot + (uint32_t)((idx & 1) * ITEM_BYTES + 16 * lane),
                           reinterpret_cast<const uint8_t*>(my_items + idx) + 16 * lane);
        };
        if (FORM == BATCHED && my_tiles > 0) fetch_item(0);
        wait_for_operands();
        for (int i = 0; ok && i < my_tiles; i++) {
            // batched: the drain takes what it needs of the work item, the rest is
            // read after it, so that the drained columns have the registers
            const TcWorkItem* w =
                reinterpret_cast<const TcWorkItem*>(smem + (islot - sbase) + (i & 1) * ITEM_BYTES);
            Tile tc;
            if (FORM == BATCHED) {
                cp_async_wait_all();
                __syncwarp();
                if (i + 1 < my_tiles) fetch_item(i + 1);
                tc.nvec = w->nks;
                tc.op = w->op;
                tc.n128 = w->n128;
            } else {
                tc = get_tile<FORM>(p, my_items, i, &tmA, &tmB);
            }
            const int nst = (tc.nvec + STAGE_VECS - 1) / STAGE_VECS;
            const int chunk = chunk_of(tc.op);
            const int nseg = (nst + chunk - 1) / chunk;
            const bool gf2 = tc.op == OP_GF2;
            const bool idle = tc.n128 && chalf == 1;
            uint32_t words[CW];
#pragma unroll
            for (int c = 0; c < CW; c++) words[c] = 0u;
            for (int g = 0; g < nseg; g++, seg++) {
                if (!warp_wait(acc_full, seg & 1, p.err)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                if (idle) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(acc_empty, 0);
                    continue;
                }
                // everything this warp drains is in registers before it packs, so
                // the accumulator goes back at once
                uint32_t v[64];
                tmem_ld128_low(tlane + (uint32_t)(128 * chalf), v);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(acc_empty, 0);
                if (gf2) {
#pragma unroll
                    for (int c = 0; c < CW; c++) words[c] ^= pack_low<OP_GF2>(v + 16 * c);
                } else {
#pragma unroll
                    for (int c = 0; c < CW; c++) words[c] |= pack_low<OP_BOOL>(v + 16 * c);
                }
            }
            if (!ok) break;
            if (FORM == BATCHED) tc = item_tile(p, *w);
            const int64_t row = (int64_t)tc.tm * TILE_M + (int64_t)rank * BM + 32 * quarter + lane;
            if (row < tc.m) {
                uint64_t* crow = tc.C + row * tc.ldc;
                const int64_t w0 = (int64_t)tc.tn * (BN / 64) + chalf * (CW / 2);
                const int64_t nw = tc.n / 64;
                if (FORM == SLICED && tc.nvec != p.nvec) {
#pragma unroll
                    for (int c = 0; c < CW / 2; c++) {
                        const uint64_t w = (uint64_t)words[2 * c] | ((uint64_t)words[2 * c + 1] << 32);
                        if (w0 + c < nw) {
                            if (gf2)
                                red_xor(crow + w0 + c, w);
                            else
                                red_or(crow + w0 + c, w);
                        }
                    }
                } else if (w0 + 1 < nw && (reinterpret_cast<uintptr_t>(crow) & 15) == 0) {
                    *reinterpret_cast<uint4*>(crow + w0) =
                        make_uint4(words[0], words[1], words[2], words[3]);
                } else {
#pragma unroll
                    for (int c = 0; c < CW / 2; c++)
                        if (w0 + c < nw)
                            crow[w0 + c] = (uint64_t)words[2 * c] | ((uint64_t)words[2 * c + 1] << 32);
                }
            }
        }
        // a loop left early (a wait gave up) may still have an item copy in
        // flight into this warp's slot
        if (FORM == BATCHED) cp_async_wait_all();
    } else if (warp == TMA_WARP) {
        // ---------------------------------------------------- TMA producer
        // The whole warp runs the loop and one elected lane issues: from a lane
        // of a divergent warp the two copies of a stage take 450 cycles to issue,
        // which is most of the 512 that the stage's MMAs take.
        int st = 0;  // stages issued
        int s = 0;   // the next one's place
        uint32_t s_parity = 1;
        bool ok = true;
        // Batched: a tile's work item is read two tiles ahead and its
        // TMA maps prefetched one tile ahead.
        Tile nxt = my_tiles > 0 ? get_tile<FORM>(p, my_items, 0, &tmA, &tmB) : Tile{};
        Tile nxt2 = my_tiles > 1 ? get_tile<FORM>(p, my_items, 1, &tmA, &tmB) : nxt;
        if (FORM == BATCHED && my_tiles > 0 && elect_one()) {
            prefetch_tensormap(nxt.ma);
            prefetch_tensormap(nxt.mb);
        }
        wait_for_operands();
        for (int i = 0; ok && i < my_tiles; i++) {
            const Tile tc = nxt;
            nxt = nxt2;
            if (FORM == BATCHED && i + 1 < my_tiles && elect_one()) {
                prefetch_tensormap(nxt.ma);
                prefetch_tensormap(nxt.mb);
            }
            if (i + 2 < my_tiles) nxt2 = get_tile<FORM>(p, my_items, i + 2, &tmA, &tmB);
            const int arow = tc.tm * TILE_M + (int)rank * BM;
            // an N = 128 tile takes 64 of its columns from each CTA
            const int brow = tc.tn * BN + (int)rank * (tc.n128 ? BROWS / 2 : BROWS);
            const int v0 = FORM == SLICED ? tc.leaf : 0;
            const int leaf = FORM == SLICED ? 0 : tc.leaf;
            for (int v = v0; v < v0 + tc.nvec; v += STAGE_VECS, st++) {
                if (!warp_wait(empty_p(s), s_parity, p.err)) {
                    ok = false;
                    break;
                }
                if (elect_one()) {
                    // (its readers see it through the barrier)
                    *reinterpret_cast<volatile uint32_t*>(smem + OFF_SKIP + 4 * s) = 16u * (v & 1);
                    mbar_arrive_tx(full_p(s), PA_BYTES + PB_BYTES);
                    const int word = 2 * v & ~3;
                    tma_load_3d(sbase + OFF_PA + s * PA_BYTES, tc.ma, word, arow, leaf,
                                full_p(s));
                    tma_load_3d(sbase + OFF_PB + s * PB_BYTES, tc.mb, word, brow, leaf,
                                full_p(s));
                }
                __syncwarp();
                if (++s == PSTAGES) {
                    s = 0;
                    s_parity ^= 1;
                }
            }
        }
        // drain: the copies of the last issued stages must land before exit
        for (int j = 1; j <= PSTAGES && j <= st; j++) {
            const int i = st - j;
            if (!warp_wait(full_p(i % PSTAGES), (i / PSTAGES) & 1, p.err)) break;
        }
    } else if (warp == MMA_WARP && rank == 0) {
        // ---------------------------------------------------- MMA issuer
        const uint64_t db_base = smem_desc_plain(sbase + OFF_EB);
        const uint64_t bias_desc = smem_desc_plain(sbase + OFF_BIAS);
        int seg = 0;
        uint32_t st = 0;  // running stage count
        bool ok = true;
        uint32_t seen = 0;  // this packed stage's operands have been seen ready
        TileK nxt = my_tiles > 0 ? get_tile_k<FORM>(p, my_items, 0) : TileK{0, 0, 1};
        TileK nxt2 = my_tiles > 1 ? get_tile_k<FORM>(p, my_items, 1) : nxt;
        wait_for_operands();
        for (int i = 0; ok && i < my_tiles; i++) {
            const int nvec = nxt.nvec, chunk = nxt.chunk;
            const uint32_t id = nxt.n128 ? instr_desc_k96<BN / 2>() : instr_desc_k96<BN>();
            nxt = nxt2;
            if (i + 2 < my_tiles) nxt2 = get_tile_k<FORM>(p, my_items, i + 2);
            int kin = 0;  // stages in the accumulator
            for (int left = nvec; left > 0; left -= STAGE_VECS, st++) {
                // At a tile's first slot the operands are checked before the
                // (longer) wait for the epilogue to free the accumulator.
                if (!__all_sync(0xffffffffu, seen) &&
                    !warp_wait(full_o(st & (SLOTS - 1)), (st / SLOTS) & 1u, p.err)) {
                    ok = false;
                    break;
                }
                if (kin == 0 && !warp_wait(acc_empty, (seg & 1) ^ 1, p.err)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                // the next slot's barrier is read while this one's MMAs go out
                seen = mbar_test(full_o((st + 1) & (SLOTS - 1)), ((st + 1) / SLOTS) & 1u);
                constexpr uint64_t STEP = 3 * CHUNK_BYTES >> 4;
                const uint32_t q = st & (SLOTS - 1);
                const uint32_t ta = A_COL + q * SLOT_COLS;
                const uint64_t db = db_base + (uint64_t)(q * (EB_BYTES >> 4));
                // One block of code for every stage: v vectors of 128 bits take v + 1
                // MMAs, and with the last stage the counts leave the accumulator.
                const bool ends = left <= STAGE_VECS || kin + 1 >= chunk;
                if (elect_one()) {
                    if (kin == 0) mma_k96<BIAS>(BIAS_A_COL, bias_desc, id);
                    mma_k96<KINDS>(ta, db, id);
                    if (left > 1) mma_k96<KINDS>(ta + MMA_COLS, db + STEP, id);
                    if (left > 2) mma_k96<KINDS>(ta + 2 * MMA_COLS, db + 2 * STEP, id);
                    mma_k96<ONES>(ta + 3 * MMA_COLS, db + 3 * STEP, id);
                    mma_commit<true>(empty_o(q));
                    if (ends) mma_commit<true>(acc_full);
                }
                __syncwarp();
                kin = ends ? 0 : kin + 1;
                seg += ends;
            }
        }
        if (!ok) {  // wait (bounded) for every MMA issued so far
            if (elect_one()) mma_commit<true>(drain_bar, 1);
            __syncwarp();
            warp_wait(drain_bar, 0, p.err);
        }
    }

    tc_fence_before();
    __syncthreads();
    // A pair leaves together: the peer's remote arrivals and the MMAs that
    // read its shared memory and TMEM are over before either CTA frees TMEM.
    cluster_sync();
    if (warp == MMA_WARP) {
        tc_fence_after();
        tmem_dealloc<true>(0u);
    }
}

// ---------------------------------------------------------------- host side
constexpr int MAX_DEVICES = 64;
std::mutex g_setup_mu;

template <int FORM>
cudaError_t set_smem_attr(int d) {
    static bool done[MAX_DEVICES] = {false};
    static cudaError_t err[MAX_DEVICES];
    std::lock_guard<std::mutex> lk(g_setup_mu);
    if (!done[d]) {
        err[d] = cudaFuncSetAttribute(tc_fp4_kernel<FORM>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
        done[d] = true;
    }
    return err[d];
}

int device_index() {
    int d = -1;
    return cudaGetDevice(&d) == cudaSuccess && d >= 0 && d < MAX_DEVICES ? d : -1;
}

cudaLaunchConfig_t pair_config(unsigned units, cudaLaunchAttribute* at) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * units);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cfg;
}

template <int FORM>
cudaError_t launch(const CUtensorMap& ma, const CUtensorMap& mb, const Params& prm, int units,
                   cudaStream_t s) {
    const int d = device_index();
    if (d < 0) return cudaErrorInvalidDevice;
    const cudaError_t e = set_smem_attr<FORM>(d);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at[2];
    cudaLaunchConfig_t cfg = pair_config((unsigned)units, at);
    cfg.stream = s;
    return cudaLaunchKernelEx(&cfg, tc_fp4_kernel<FORM>, ma, mb, prm);
}

}  // namespace

// CTA pairs that can be resident at once (clusters of two on one TPC); 0 if
// cluster launches are unavailable.
int tc_fp4_slots() {
    static int slots[MAX_DEVICES];
    static bool done[MAX_DEVICES] = {false};
    const int d = device_index();
    if (d < 0 || set_smem_attr<WHOLE>(d) != cudaSuccess) return 0;
    std::lock_guard<std::mutex> lk(g_setup_mu);
    if (!done[d]) {
        cudaLaunchAttribute at[2];
        const cudaLaunchConfig_t cfg = pair_config((unsigned)sm_count(), at);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, tc_fp4_kernel<WHOLE>, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            n = 0;
        }
        slots[d] = n;
        done[d] = true;
    }
    return slots[d];
}

bool tc_fp4_maps(CUtensorMap* ma, CUtensorMap* mb, const uint64_t* A, int64_t lda, int64_t strideA,
                 const uint64_t* Bt, int64_t ldb, int64_t strideB, int64_t count, int64_t m,
                 int64_t k, int64_t n) {
    return tc_make_map(ma, A, k / 64, m, lda, count, strideA, BM, ROW_BYTES / 8, true) &&
           tc_make_map(mb, Bt, k / 64, n, ldb, count, strideB, BROWS, ROW_BYTES / 8, true);
}

// The tiles past the last full round of units, where they fill less than half of
// them, are cut along k into as many slices as there are units for each. A slice
// costs C's zeros beforehand, the start of an accumulator and reductions into C, so
// the longest has to be at least MIN_SAVED stages shorter than the tile. Measured
// (us inside a graph, whole -> sliced): less than half a round in all, 64 x 32768 x
// 64 28.1 -> 6.7, 512 x 32768 x 512 30.5 -> 10.1, 192 x 12288 x 4096 17.1 -> 12.1,
// 512 x 4096 x 512 10.0 -> 7.2; after full rounds, 2112 x 1984 x 2240 10.9 -> 10.1,
// 4096^3 21.0 -> 20.3, 8192^3 99.5 -> 96, 8192 x 1984 x 8192 38.2 -> 35.6. Where
// three stages are all that is saved it can lose 3 % (2816 x 1984 x 2560 10.97 ->
// 11.3) or gain 8 % (4096 x 2048 x 4096 15.6 -> 14.4).
int tc_fp4_slice_stages(int64_t m, int64_t k, int64_t n, TileRange* zero) {
    constexpr int MIN_SAVED = 3;
    const int64_t slots = tc_fp4_slots();
    const int64_t tm = (m + TILE_M - 1) / TILE_M, tn = (n + BN - 1) / BN;
    if (slots <= 0 || slots > 255 || tm * tn > 0x7fffffff || k > 0x7fffffff) return 0;
    const int64_t tail = tm * tn % slots;
    if (tail == 0 || 2 * tail > slots) return 0;
    const int64_t stages = (k + 128 * STAGE_VECS - 1) / (128 * STAGE_VECS);
    const int64_t slices = slots / tail;
    const int64_t each = (stages + slices - 1) / slices;
    if (stages - each < MIN_SAVED) return 0;
    if (zero) {
        zero->first = (int)(tm * tn - tail);
        zero->count = (int)tail;
        zero->order.set((int)tm, (int)tn);
    }
    return (int)each;
}

bmm_status run_fp4_strided(int op, const uint64_t* A, int64_t lda, int64_t strideA,
                           const uint64_t* Bt, int64_t ldb, int64_t strideB, uint64_t* C,
                           int64_t ldc, int64_t strideC, int64_t count, int64_t m, int64_t k,
                           int64_t n, cudaStream_t s, int slice_stages) {
    const int slots = tc_fp4_slots();
    if (slots <= 0) return BMM_ERR_UNSUPPORTED;
    uint32_t* err = device_error_word();
    if (!err) return BMM_ERR_NOMEM;
    CUtensorMap ma, mb;
    if (!tc_fp4_maps(&ma, &mb, A, lda, strideA, Bt, ldb, strideB, count, m, k, n))
        return BMM_ERR_CUDA;
    Params prm{};
    prm.C = C;
    prm.ldc = ldc;
    prm.strideC = strideC;
    prm.m = (int)m;
    prm.n = (int)n;
    prm.nvec = (int)((k + 127) / 128);
    prm.op = op;
    const int64_t tiles_m = (m + TILE_M - 1) / TILE_M, tiles_n = (n + BN - 1) / BN;
    const int64_t total = tiles_m * tiles_n * count;
    if (total > 0x7fffffff) return BMM_ERR_UNSUPPORTED;
    prm.order.set((int)tiles_m, (int)tiles_n);
    prm.items_total = (int)total;
    if (slice_stages > 0) {
        const int64_t vecs = slice_stages * STAGE_VECS, tail = total % slots;
        const int64_t slices = tail * ((prm.nvec + vecs - 1) / vecs);
        if (count > 1 || tail == 0 || slices > slots || slots > 255) return BMM_ERR_INVALID;
        prm.whole = (int)(total - tail);
        prm.items_total = prm.whole + (int)slices;
        prm.strideC = vecs | ((65535 + tail) / tail) << 32;
    }
    prm.err = err;
    TraceScope ts(BMM_PHASE_BASE, s);
    const int units = prm.items_total < slots ? prm.items_total : slots;
    const cudaError_t e = slice_stages > 0 ? launch<SLICED>(ma, mb, prm, units, s)
                                           : launch<WHOLE>(ma, mb, prm, units, s);
    return e == cudaSuccess ? BMM_OK : cuda_fail(e);
}

cudaError_t tc_fp4_prepare_batched() {
    const int d = device_index();
    return d < 0 ? cudaErrorInvalidDevice : set_smem_attr<BATCHED>(d);
}

cudaError_t tc_fp4_launch_batched(const TcProblem* d_probs, const TcWorkItem* d_items,
                                  const int32_t* d_unit_ptr, int units, cudaStream_t s) {
    uint32_t* err = device_error_word();
    if (!err) return cudaErrorMemoryAllocation;
    Params prm{};
    prm.probs = d_probs;
    prm.items = d_items;
    prm.unit_ptr = d_unit_ptr;
    prm.err = err;
    CUtensorMap none;
    std::memset(&none, 0, sizeof(none));
    TraceScope ts(BMM_PHASE_BASE, s);
    return launch<BATCHED>(none, none, prm, units, s);
}

}  // namespace bmm
