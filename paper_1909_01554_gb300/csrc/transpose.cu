// Bit-matrix transpose (Sec. 3.5: the paper transposes the right operand so
// that both operands of the inner product run along k; it does this on the
// host with recursive word transposes) and, in the same launch, the copy of a
// left operand into rows of an even number of words. Here: on the GPU, one
// thread per 32 x 32 bit block, the recursive block swap done in its registers.
//
// A CTA moves a tile of 512 x 512 bits (256 x 512 in a batch). Thread (rb, c)
// loads word c of the 32 rows of row block rb (16 lanes read a row's 64 bytes),
// transposes the block in 256 instructions (two steps of byte permutes, three of
// shifts and LOP3), and leaves it in shared memory in the place it has in the
// output tile, from where 8 lanes (4 in a batch) write a row's words.
//
// What bounds it: a small matrix is one tile's chain of latencies (launch,
// load, store), a large one the L2 and HBM traffic of its rows*cols/8 bytes
// each way. 64 x 64 blocks swapped with shuffles took five times the
// instructions (7.5 us for a tile alone), and TMA boxes in the place of these
// loads and stores were slower at every size. Measured inside a graph (us): 512 x
// 512 3.0, 4096 x 4096 3.3, 16384 x 16384 11.2, 32768 x 32768 44.8 (6.0 TB/s; 48.3
// with 64-bit offsets), 32704 x 32704 48.8 (rows that start at odd 8-byte places
// touch three sectors for two), 65536 x 65536 170 (6.3 TB/s); back to back on
// matrices that L2 does not hold, 16448 x 12224 12.5 (4.0 TB/s). The copy in the same
// launch saves a product with k / 64 odd two memsets and a 2-D copy, a batch a
// launch.
#include "internal.h"
#include "pdl.cuh"
#include "transpose32.cuh"

namespace bmm {
namespace {

// A tile: ROWS of X's rows by TILE_COLS of its columns. ROWS = 512 for a launch's own
// matrix; 256 for a batch's, of many sizes, whose many small matrices fill more of the
// smaller tiles: 512 products of sides 64-768 26.4 us against 27.8, 256 of sides
// 256-8192 810 against 821 (as calls). A large matrix alone is faster in the larger
// tile (32768 x 32768 45 us against 47, odd output pitches 51 against 66); a small one
// is faster in the smaller (4096 x 4096 3.1 against 2.6), yet not the product behind it
// (Boolean 2112 x 1984 x 2240 10.2 against 10.3, 16384 x 12288 x 192 16.2 against 16.5).
// 256 x 256 is slower than both at size.
constexpr int TILE_COLS = 512;
constexpr int BLOCK_COLS = TILE_COLS / 32;
template <int ROWS>
struct Tile {
    static constexpr int W32 = ROWS / 32;  // 32-bit words of an output row, row blocks
    static constexpr int W64 = ROWS / 64;
    static constexpr int THREADS = W32 * BLOCK_COLS;
    static constexpr int LINE = 32 / W32;  // output rows over the 32 banks
    // Copied words per CTA (rows are never split): 8 a thread. With 16 Boolean 2112 x
    // 1984 x 2240 takes 11.4 us for 10.2 and 512 small products 27.3 for 26.3; with 4
    // 256 products of sides 256-8192 814 for 803.
    static constexpr int64_t COPY_WORDS = 8 * THREADS;

    // Word offset of 32-bit word w of output row r in the shared tile. Words are
    // rotated by two per 32 rows and rows swapped within their LINE, another way in
    // each LINE-th part of the tile, so that both the stores (lanes over 16 column blocks
    // and two words) and the 8-byte loads (lanes over rows) fall on 32 different banks.
    __device__ static __forceinline__ int at(int r, int w) {
        return ((r ^ (r / (TILE_COLS / LINE) & (LINE - 1))) * W32) + ((w + 2 * (r >> 5)) & (W32 - 1));
    }
};

// Tile (bx, by) of X^T: input rows from ROWS by, columns from 512 bx. Sizes are
// multiples of 64, so every 32 x 32 block lies wholly inside or outside. Rows
// past X's count as zero, up to the output's row pitch. Offset holds the bytes from
// a tile's corner to any of its words: with 32 bits a word's address is one
// addition to the CTA's base.
template <int ROWS, typename Offset>
__device__ __forceinline__ void transpose_tile(const TransposeJob& j, uint32_t bx, uint32_t by,
                                               uint32_t* tile) {
    using T = Tile<ROWS>;
    const int t = threadIdx.x;
    const int64_t r0 = (int64_t)by * ROWS, c0 = (int64_t)bx * TILE_COLS;
    const int cols = (int)(j.cols - c0 < TILE_COLS ? j.cols - c0 : TILE_COLS);
    {
        const char* src = reinterpret_cast<const char*>(j.X + r0 * j.pitch + c0 / 64);
        const int c = t & (BLOCK_COLS - 1), rb = t / BLOCK_COLS;
        const Offset step = (Offset)(8 * j.pitch), at = 32 * rb * step + 4 * c;
        uint32_t v[32];
        if (r0 + 32 * rb < j.rows && 32 * c < cols) {
#pragma unroll
            for (int i = 0; i < 32; i++) v[i] = *reinterpret_cast<const uint32_t*>(src + (at + i * step));
            transpose32(v);
        } else {
#pragma unroll
            for (int i = 0; i < 32; i++) v[i] = 0u;
        }
#pragma unroll
        for (int l = 0; l < T::LINE; l++) {
            uint32_t* at_l = tile + T::at(32 * c + l, rb);
#pragma unroll
            for (int i = l; i < 32; i += T::LINE) at_l[(i - l) * T::W32] = v[i];
        }
    }
    __syncthreads();
    const int q = t & (T::W64 - 1), r = t / T::W64;
    if ((int64_t)by * T::W64 + q >= j.tpitch) return;
    static_assert(T::THREADS == 32 * T::W64, "32 output rows a step");
    char* dst = reinterpret_cast<char*>(j.Xt + c0 * j.tpitch + r0 / 64);
    const Offset step = (Offset)(8 * 32 * j.tpitch), at = r * (Offset)(8 * j.tpitch) + 8 * q;
#pragma unroll
    for (int s = 0; s < BLOCK_COLS; s++)
        if (32 * s < cols)
            *reinterpret_cast<uint64_t*>(dst + (at + s * step)) =
                *reinterpret_cast<const uint64_t*>(tile + T::at(32 * s + r, 2 * q));
}

template <int ROWS>
__host__ __device__ inline int64_t copy_rows(int64_t tpitch) {
    return tpitch >= Tile<ROWS>::COPY_WORDS ? 1 : Tile<ROWS>::COPY_WORDS / tpitch;
}

template <int ROWS>
int64_t units_of(const TransposeJob& j) {
    if (j.copy) {
        const int64_t r = copy_rows<ROWS>(j.tpitch);
        return (j.rows + r - 1) / r;
    }
    constexpr int W64 = Tile<ROWS>::W64;
    return ((j.cols + TILE_COLS - 1) / TILE_COLS) * ((j.tpitch + W64 - 1) / W64);
}

// Rows [unit * R, ...) of Y: X's pitch words, then zeros up to Y's pitch.
template <int ROWS>
__device__ __forceinline__ void copy_unit(const TransposeJob& j, int64_t unit) {
    constexpr int THREADS = Tile<ROWS>::THREADS;
    const int64_t R = copy_rows<ROWS>(j.tpitch), r0 = unit * R;
    const int64_t rows = j.rows - r0 < R ? j.rows - r0 : R;
    const uint64_t* src = j.X + r0 * j.pitch;
    uint64_t* dst = j.Xt + r0 * j.tpitch;
    if (R == 1) {
        for (int64_t w = threadIdx.x; w < j.tpitch; w += THREADS) dst[w] = w < j.pitch ? src[w] : 0ull;
        return;
    }
    const uint32_t kp = (uint32_t)j.tpitch, kw = (uint32_t)j.pitch, words = (uint32_t)rows * kp;
    for (uint32_t i = threadIdx.x; i < words; i += THREADS) {
        const uint32_t r = i / kp, w = i - r * kp;
        dst[i] = w < kw ? src[r * kw + w] : 0ull;
    }
}

template <int ROWS, typename Offset>
__device__ __forceinline__ void run_unit(const TransposeJob& j, uint32_t unit) {
    __shared__ __align__(16) uint32_t tile[TILE_COLS * Tile<ROWS>::W32];
    if (j.copy) {
        copy_unit<ROWS>(j, unit);
        return;
    }
    // Tiles below one another first, so the output is written by whole rows. Where
    // its rows start at odd 8-byte places two tiles write parts of one sector: 32704 x
    // 32704 takes 49 us in this order, 65 with tiles beside one another first (and in
    // groups of 4 or 16 rows of tiles). Even pitches run alike: 32768 x 32768 45 us.
    const uint32_t gy = (uint32_t)((j.tpitch + Tile<ROWS>::W64 - 1) / Tile<ROWS>::W64);
    transpose_tile<ROWS, Offset>(j, unit / gy, unit % gy, tile);
}

// Job a takes the first `split` CTAs, job b those before `zeros`, the rest write
// one tile's zeros each.
template <int ROWS, typename Offset>
__global__ void __launch_bounds__(Tile<ROWS>::THREADS)
    prepare_kernel(const TransposeJob a, const TransposeJob b, const ZeroJob z, uint32_t split,
                   uint32_t zeros) {
    wait_for_operands();
    dependents_may_launch();
    const uint32_t u = blockIdx.x;
    if (u >= zeros) {
        static_assert(Tile<ROWS>::THREADS == 256, "a thread a row of the tile");
        const TileCoord c = z.tiles.order.tile(z.tiles.first + (int)(u - zeros));
        const int64_t row = (int64_t)c.tm * 256 + threadIdx.x, w0 = (int64_t)c.tn * 4;
        if (row < z.m)
            for (int64_t w = w0; w < w0 + 4 && w < z.n / 64; w++) z.C[row * z.ldc + w] = 0ull;
        return;
    }
    run_unit<ROWS, Offset>(u < split ? a : b, u < split ? u : u - split);
}

// Many jobs in one launch: CTA b takes unit b - first[i] of job i = job_of[b] (a
// table: a search through first[] would be some ten loads one after the other).
template <int ROWS, typename Offset>
__global__ void __launch_bounds__(Tile<ROWS>::THREADS)
    prepare_batched_kernel(const TransposeJob* __restrict__ jobs, const int64_t* __restrict__ first,
                           const int32_t* __restrict__ job_of) {
    const int32_t i = job_of[blockIdx.x];
    const TransposeJob j = jobs[i];
    const uint32_t unit = (uint32_t)(blockIdx.x - first[i]);
    wait_for_operands();
    dependents_may_launch();
    run_unit<ROWS, Offset>(j, unit);
}

constexpr int ONE = 512, MANY = 256;  // tile rows of the two forms

}  // namespace

bool prepare_far(const TransposeJob& j) {
    constexpr int64_t NEAR = (1ll << 32) / (8 * 512);
    return !j.copy && (j.pitch >= NEAR || j.tpitch >= NEAR);
}

int64_t prepare_units(const TransposeJob& j) { return units_of<MANY>(j); }

cudaError_t launch_prepare(const TransposeJob& j, const TransposeJob* copy, const ZeroJob& zero,
                           cudaStream_t s) {
    const int64_t tiles = units_of<ONE>(j), zeros = tiles + (copy ? units_of<ONE>(*copy) : 0);
    const int64_t units = zeros + zero.tiles.count;
    // (the callers' limit on rows, 65535 tiles, is kept though the grid has no such one)
    if ((j.rows + ONE - 1) / ONE > 65535 || units > 0x7fffffff)
        return cudaErrorInvalidConfiguration;
    if (units <= 0) return cudaSuccess;
    TraceScope ts(BMM_PHASE_TRANSPOSE, s);
    return launch_pdl(prepare_far(j) ? prepare_kernel<ONE, uint64_t> : prepare_kernel<ONE, uint32_t>,
                      dim3((unsigned)units), Tile<ONE>::THREADS, 0, s, j, copy ? *copy : j, zero,
                      (uint32_t)tiles, (uint32_t)zeros);
}

cudaError_t launch_prepare_batched(const TransposeJob* jobs, const int64_t* first,
                                   const int32_t* job_of, int64_t total_units, bool far,
                                   cudaStream_t s) {
    if (total_units <= 0) return cudaSuccess;
    if (total_units > 0x7fffffff) return cudaErrorInvalidConfiguration;
    TraceScope ts(BMM_PHASE_TRANSPOSE, s);
    return launch_pdl(far ? prepare_batched_kernel<MANY, uint64_t> : prepare_batched_kernel<MANY, uint32_t>,
                      dim3((unsigned)total_units), Tile<MANY>::THREADS, 0, s, jobs, first, job_of);
}

}  // namespace bmm
