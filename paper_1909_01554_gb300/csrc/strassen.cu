// XOR passes of the Strassen-like recursions over packed words: basis changes
// (Secs. 3.6 and 3.13), the expanding parallel layer (Sec. 3.9, Alg. 1), the
// compressing parallel layer (Sec. 3.11, Alg. 2) with up to two levels merged
// in registers (Sec. 3.15), and the depth-first combine / fold passes of the
// serial layer (Sec. 3.8, Eqs. rec-in and rec-out).
//
// All are HBM-bound streaming kernels: one thread per 64-bit word position of
// the leaf-sized block, coalesced along the row, every input word read once
// and every output word written once.
#include "internal.h"
#include "pdl.cuh"
#include "plan.h"
#include "slp.h"
#include "tile_order.h"

namespace bmm {
namespace {

// Stored block (r, c) of an operand for block index q = 2*i + j of the paper's
// operand. The right operand is held transposed (Bt = B^T), so block (j, k)
// of B is the transpose of stored block (k, j).
template <int OPERAND>
__device__ __forceinline__ void stored_block(int q, int& r, int& c) {
    if (OPERAND == 0) {
        r = q >> 1;
        c = q & 1;
    } else {
        r = q & 1;
        c = q >> 1;
    }
}

// The blocks an expanding pass reads: the block X itself (mask 0), or the
// quadrants `mask` selects of the parent block X of twice the size, XORed
// together (the input combination of a depth-first level, Eq. rec-in, fused
// into the pass). Returns how many, with their offsets in words from X;
// brows x bw is the expanded block's size in words.
template <int OPERAND>
__device__ __forceinline__ int source_blocks(uint32_t mask, int64_t pitch, int64_t brows,
                                             int64_t bw, int64_t (&off)[4]) {
    if (mask == 0) {
        off[0] = 0;
        return 1;
    }
    int cnt = 0;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        if (!((mask >> q) & 1u)) continue;
        int r, c;
        stored_block<OPERAND>(q, r, c);
        off[cnt++] = r * brows * pitch + c * bw;
    }
    return cnt;
}

// The blocks a compressing pass writes: C itself (dest 0), or the quadrants
// `dest` selects of the parent C (the output fold of a depth-first level,
// Eq. rec-out, fused into the pass): block q becomes v where bit q of
// `first` is set, else is XORed with v.
__device__ __forceinline__ int dest_blocks(uint32_t dest, uint32_t first, int64_t ldc,
                                           int64_t brows, int64_t bw, int64_t (&off)[4],
                                           bool (&overwrite)[4]) {
    if (dest == 0) {
        off[0] = 0;
        overwrite[0] = true;
        return 1;
    }
    int cnt = 0;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        if (!((dest >> q) & 1u)) continue;
        off[cnt] = (q >> 1) * brows * ldc + (q & 1) * bw;
        overwrite[cnt++] = (first >> q) & 1u;
    }
    return cnt;
}

// A position's row: t / width, by a multiplication where t is below 2^31 (the 64-bit
// division takes more instructions than the rest of a one-level pass).
__device__ __forceinline__ int64_t row_of(int64_t t, int64_t width, const FastDiv& div) {
    return t <= 0x7fffffff ? (int64_t)div((uint32_t)t) : t / width;
}
FastDiv divide_by(int64_t width) {
    FastDiv d;
    d.set((uint32_t)(width <= 0x7fffffff ? width : 1));
    return d;
}

template <int V, int OPERAND, typename Wd>
__device__ __forceinline__ void combine_level(const Wd* in, Wd* out) {
    if (OPERAND == 0)
        slp::alpha<V>(in, out);
    else
        slp::beta<V>(in, out);
}

// One operand of an expanding pass: rows x wcols is the expanded block; with a
// non-zero mask it is formed on the fly from its parent X (source_blocks).
struct ExpandJob {
    const uint64_t* X;
    uint64_t* leaves;
    int64_t pitch, rows, wcols;
    uint32_t mask;
    FastDiv width;  // of a leaf in words
};

// Expanding pass over D merged levels: basis change (phi / psi) then the
// operand combinations (alpha / beta) at every level, from 4^D input words
// to 7^D leaf words per position. Leaf index H = h_1 7^(D-1) + ... + h_D
// (level 1 most significant). `blocks` CTAs, of which this is `block`.
template <int V, int D, int OPERAND>
__device__ __forceinline__ void expand(const ExpandJob& j, int64_t block, int64_t blocks) {
    const uint64_t* X = j.X;
    uint64_t* __restrict__ leaves = j.leaves;
    const int64_t pitch = j.pitch;
    const int64_t lr = j.rows >> D, lw = j.wcols >> D;
    const int64_t leaf_words = lr * lw;
    const int64_t total = leaf_words;
    int64_t soff[4];
    const int nsrc = source_blocks<OPERAND>(j.mask, pitch, j.rows, j.wcols, soff);
    for (int64_t t = block * blockDim.x + threadIdx.x; t < total; t += blocks * blockDim.x) {
        const int64_t i = row_of(t, lw, j.width), w = t - i * lw;
        if (D == 1) {
            uint64_t x[4] = {0, 0, 0, 0}, y[7];
            for (int u = 0; u < nsrc; u++) {
                const uint64_t* src = X + soff[u];
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    int r, c;
                    stored_block<OPERAND>(q, r, c);
                    x[q] ^= src[(r * lr + i) * pitch + c * lw + w];
                }
            }
            slp::phi<V>(x);
            combine_level<V, OPERAND>(x, y);
#pragma unroll
            for (int h = 0; h < 7; h++) leaves[h * leaf_words + t] = y[h];
        } else {
            uint64_t x[4][4];  // [level-1 block][level-2 block]
#pragma unroll
            for (int q1 = 0; q1 < 4; q1++)
#pragma unroll
                for (int q2 = 0; q2 < 4; q2++) x[q1][q2] = 0;
            for (int u = 0; u < nsrc; u++) {  // 16 independent loads per source block
                const uint64_t* src = X + soff[u];
#pragma unroll
                for (int q1 = 0; q1 < 4; q1++)
#pragma unroll
                    for (int q2 = 0; q2 < 4; q2++) {
                        int r1, c1, r2, c2;
                        stored_block<OPERAND>(q1, r1, c1);
                        stored_block<OPERAND>(q2, r2, c2);
                        x[q1][q2] ^= src[(r1 * 2 * lr + r2 * lr + i) * pitch + c1 * 2 * lw +
                                         c2 * lw + w];
                    }
            }
            // basis change at level 2 (within each level-1 block) and at level 1
#pragma unroll
            for (int q1 = 0; q1 < 4; q1++) slp::phi<V>(x[q1]);
#pragma unroll
            for (int q2 = 0; q2 < 4; q2++) {
                uint64_t v[4] = {x[0][q2], x[1][q2], x[2][q2], x[3][q2]};
                slp::phi<V>(v);
#pragma unroll
                for (int q1 = 0; q1 < 4; q1++) x[q1][q2] = v[q1];
            }
            // level-2 combinations, then level-1 combinations (Yates)
            uint64_t y[4][7];
#pragma unroll
            for (int q1 = 0; q1 < 4; q1++) combine_level<V, OPERAND>(x[q1], y[q1]);
#pragma unroll
            for (int h2 = 0; h2 < 7; h2++) {
                uint64_t v[4] = {y[0][h2], y[1][h2], y[2][h2], y[3][h2]}, z[7];
                combine_level<V, OPERAND>(v, z);
#pragma unroll
                for (int h1 = 0; h1 < 7; h1++) leaves[(h1 * 7 + h2) * leaf_words + t] = z[h1];
            }
        }
    }
}

// Both operands in one launch: the first `split` CTAs take A, the rest Bt.
// Small passes are latency (4 us each at 8192 x 4096), so one launch saves one of
// them: with it and row_of for the divisions, us a product inside a graph, 1024^3
// depth 1 12.6 -> 11.2, 2048^3 depth 2 19.1 -> 15.8, 8192^3 depth 1 107.7 -> 104.9
// and depth 2 116.3 -> 112.2, 8192 x 4096 x 8192 depth 1 69.8 -> 67.7.
template <int V, int D>
__global__ void __launch_bounds__(256, 2) expand_kernel(const ExpandJob a, const ExpandJob b,
                                                        uint32_t split) {
    wait_for_operands();
    dependents_may_launch();
    if (blockIdx.x < split)
        expand<V, D, 0>(a, blockIdx.x, split);
    else
        expand<V, D, 1>(b, blockIdx.x - split, gridDim.x - split);
}

// Compressing pass over D merged levels: gamma then the inverse basis change
// chi at every level, from 7^D leaf products to 4^D output words, written
// into C or folded into its parent (dst_word).
template <int V, int D>
__global__ void __launch_bounds__(256, 2) compress_kernel(const uint64_t* leaves,
                                                       int64_t lr, int64_t lw,
                                                       uint64_t* C, int64_t ldc,
                                                       uint32_t dest, uint32_t first,
                                                       const FastDiv width) {
    wait_for_operands();
    dependents_may_launch();
    const int64_t leaf_words = lr * lw;
    int64_t doff[4];
    bool over[4];
    const int ndst = dest_blocks(dest, first, ldc, lr << D, lw << D, doff, over);
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < leaf_words;
         t += (int64_t)gridDim.x * blockDim.x) {
        // (two merged levels have no registers to spare for it)
        const int64_t i = D == 1 ? row_of(t, lw, width) : t / lw, w = t - i * lw;
        if (D == 1) {
            uint64_t q[7], c[4];
#pragma unroll
            for (int h = 0; h < 7; h++) q[h] = leaves[h * leaf_words + t];
            slp::gamma<V>(q, c);
            slp::chi<V>(c);
            for (int u = 0; u < ndst; u++) {  // all old words loaded before any store
                uint64_t* dst = C + doff[u];
                uint64_t old[4] = {0, 0, 0, 0};
                if (!over[u]) {
#pragma unroll
                    for (int b = 0; b < 4; b++) old[b] = dst[((b >> 1) * lr + i) * ldc + (b & 1) * lw + w];
                }
#pragma unroll
                for (int b = 0; b < 4; b++)
                    dst[((b >> 1) * lr + i) * ldc + (b & 1) * lw + w] = old[b] ^ c[b];
            }
        } else {
            uint64_t u[7][4];  // [h1][level-2 block]
#pragma unroll
            for (int h1 = 0; h1 < 7; h1++) {
                uint64_t q[7];
#pragma unroll
                for (int h2 = 0; h2 < 7; h2++) q[h2] = leaves[(h1 * 7 + h2) * leaf_words + t];
                slp::gamma<V>(q, u[h1]);
            }
            uint64_t c[4][4];  // [level-1 block][level-2 block]
#pragma unroll
            for (int b2 = 0; b2 < 4; b2++) {
                uint64_t q[7] = {u[0][b2], u[1][b2], u[2][b2], u[3][b2], u[4][b2], u[5][b2], u[6][b2]};
                uint64_t v[4];
                slp::gamma<V>(q, v);
                slp::chi<V>(v);  // level-1 inverse basis change
#pragma unroll
                for (int b1 = 0; b1 < 4; b1++) c[b1][b2] = v[b1];
            }
#pragma unroll
            for (int b1 = 0; b1 < 4; b1++) slp::chi<V>(c[b1]);  // level-2 inverse basis change
            for (int u = 0; u < ndst; u++) {  // all old words loaded before any store
                uint64_t* dst = C + doff[u];
                uint64_t old[4][4];
#pragma unroll
                for (int b1 = 0; b1 < 4; b1++)
#pragma unroll
                    for (int b2 = 0; b2 < 4; b2++) {
                        const int64_t row = (b1 >> 1) * 2 * lr + (b2 >> 1) * lr + i;
                        const int64_t col = (b1 & 1) * 2 * lw + (b2 & 1) * lw + w;
                        old[b1][b2] = over[u] ? 0ull : dst[row * ldc + col];
                    }
#pragma unroll
                for (int b1 = 0; b1 < 4; b1++)
#pragma unroll
                    for (int b2 = 0; b2 < 4; b2++) {
                        const int64_t row = (b1 >> 1) * 2 * lr + (b2 >> 1) * lr + i;
                        const int64_t col = (b1 & 1) * 2 * lw + (b2 & 1) * lw + w;
                        dst[row * ldc + col] = old[b1][b2] ^ c[b1][b2];
                    }
            }
        }
    }
}

// Depth-first input combination (Eq. rec-in with the basis change folded in):
// dst = XOR of the blocks of X selected by `mask` (bit q = block q of the
// paper's operand; OPERAND 1 reads the transposed right operand).
template <int OPERAND>
__global__ void __launch_bounds__(256) combine_kernel(const uint64_t* X, int64_t pitch,
                                                      int64_t hr, int64_t hw, uint32_t mask,
                                                      uint64_t* dst) {
    wait_for_operands();
    dependents_may_launch();
    const int64_t total = hr * hw;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / hw, w = t - i * hw;
        uint64_t acc = 0;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            if (!((mask >> q) & 1u)) continue;
            int r, c;
            stored_block<OPERAND>(q, r, c);
            acc ^= X[(r * hr + i) * pitch + c * hw + w];
        }
        dst[t] = acc;
    }
}

// Depth-first output fold (Eq. rec-out): for each block q of C in `dest`,
// C_q = R (bit q of `first`) or C_q ^= R.
__global__ void __launch_bounds__(256) fold_kernel(const uint64_t* R, int64_t hr,
                                                   int64_t hw, uint64_t* C, int64_t ldc,
                                                   uint32_t dest, uint32_t first) {
    wait_for_operands();
    dependents_may_launch();
    const int64_t total = hr * hw;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / hw, w = t - i * hw;
        const uint64_t v = R[t];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            if (!((dest >> q) & 1u)) continue;
            uint64_t* p = C + ((q >> 1) * hr + i) * ldc + (q & 1) * hw + w;
            *p = ((first >> q) & 1u) ? v : (*p ^ v);
        }
    }
}

// One in-place basis-change level over all parent blocks at depth `level-1`.
template <int V, int INV>
__global__ void __launch_bounds__(256) basis_level_kernel(uint64_t* X, int64_t pitch,
                                                          int64_t rows, int64_t wcols, int level) {
    wait_for_operands();
    dependents_may_launch();
    const int64_t hr = rows >> level, hw = wcols >> level;
    const int64_t half_r = rows >> 1, half_w = wcols >> 1;
    const int64_t total = half_r * half_w;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t rho = t / half_w, omega = t - rho * half_w;
        const int64_t pr = rho / hr, i = rho - pr * hr;
        const int64_t pc = omega / hw, w = omega - pc * hw;
        uint64_t* base = X + (pr * 2 * hr + i) * pitch + pc * 2 * hw + w;
        uint64_t x[4];
#pragma unroll
        for (int q = 0; q < 4; q++) x[q] = base[(q >> 1) * hr * pitch + (q & 1) * hw];
        if (INV)
            slp::chi<V>(x);
        else
            slp::phi<V>(x);
#pragma unroll
        for (int q = 1; q < 4; q++) base[(q >> 1) * hr * pitch + (q & 1) * hw] = x[q];
    }
}

unsigned grid_for(int64_t items) {
    const int64_t cap = (int64_t)sm_count() * 8;
    int64_t b = (items + 255) / 256;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (unsigned)b;
}

template <int V>
cudaError_t launch_expand_v(int d, ExpandJob a, ExpandJob b, cudaStream_t s) {
    a.width = divide_by(a.wcols >> d);
    b.width = divide_by(b.wcols >> d);
    const unsigned split = grid_for((a.rows >> d) * (a.wcols >> d));
    const dim3 grid(split + grid_for((b.rows >> d) * (b.wcols >> d)));
    TraceScope ts(BMM_PHASE_XOR, s);
    return launch_pdl(d == 1 ? expand_kernel<V, 1> : expand_kernel<V, 2>, grid, 256, 0, s, a, b, split);
}

template <int V>
cudaError_t launch_compress_v(int d, const uint64_t* leaves, int64_t lr, int64_t lw, uint64_t* C,
                              int64_t ldc, uint32_t dest, uint32_t first, cudaStream_t s) {
    const unsigned g = grid_for(lr * lw);
    TraceScope ts(BMM_PHASE_XOR, s);
    cudaError_t e = cudaSuccess;
    if (d == 1)
        e = launch_pdl(compress_kernel<V, 1>, dim3(g), 256, 0, s, leaves, lr, lw, C, ldc, dest, first,
                       divide_by(lw));
    else
        e = launch_pdl(compress_kernel<V, 2>, dim3(g), 256, 0, s, leaves, lr, lw, C, ldc, dest, first,
                       divide_by(lw));
    return e;
}

}  // namespace

cudaError_t launch_expand(int variant, int d, const uint64_t* A, int64_t lda, int64_t m,
                          uint32_t amask, uint64_t* TL, const uint64_t* B, int64_t ldb, int64_t n,
                          uint32_t bmask, uint64_t* SL, int64_t kw, cudaStream_t s) {
    const ExpandJob a = {A, TL, lda, m, kw, amask, {}}, b = {B, SL, ldb, n, kw, bmask, {}};
    switch (variant) {
        case 0: return launch_expand_v<0>(d, a, b, s);
        case 1: return launch_expand_v<1>(d, a, b, s);
        default: return launch_expand_v<2>(d, a, b, s);
    }
}

cudaError_t launch_compress(int variant, int d, const uint64_t* leaves, int64_t lr, int64_t lw,
                            uint64_t* C, int64_t ldc, uint32_t dest, uint32_t first,
                            cudaStream_t s) {
    switch (variant) {
        case 0: return launch_compress_v<0>(d, leaves, lr, lw, C, ldc, dest, first, s);
        case 1: return launch_compress_v<1>(d, leaves, lr, lw, C, ldc, dest, first, s);
        default: return launch_compress_v<2>(d, leaves, lr, lw, C, ldc, dest, first, s);
    }
}

cudaError_t launch_combine(int operand, const uint64_t* X, int64_t pitch, int64_t hr, int64_t hw,
                           uint32_t mask, uint64_t* dst, cudaStream_t s) {
    const unsigned g = grid_for(hr * hw);
    TraceScope ts(BMM_PHASE_XOR, s);
    cudaError_t e = cudaSuccess;
    if (operand == 0)
        e = launch_pdl(combine_kernel<0>, dim3(g), 256, 0, s, X, pitch, hr, hw, mask, dst);
    else
        e = launch_pdl(combine_kernel<1>, dim3(g), 256, 0, s, X, pitch, hr, hw, mask, dst);
    return e;
}

cudaError_t launch_fold(const uint64_t* R, int64_t hr, int64_t hw, uint64_t* C, int64_t ldc,
                        uint32_t dest, uint32_t first, cudaStream_t s) {
    TraceScope ts(BMM_PHASE_XOR, s);
    return launch_pdl(fold_kernel, dim3(grid_for(hr * hw)), 256, 0, s, R, hr, hw, C, ldc, dest, first);
}

bmm_status run_basis_change(int variant, int inverse, uint64_t* X, int64_t pitch, int64_t rows,
                            int64_t cols, int depth, cudaStream_t s) {
    const int64_t wcols = cols / 64;
    if (variant == 0) return BMM_OK;  // standard basis: identity
    for (int level = 1; level <= depth; level++) {
        const unsigned g = grid_for((rows / 2) * (wcols / 2));
        TraceScope ts(BMM_PHASE_XOR, s);
        cudaError_t e = cudaSuccess;
        if (variant == 1) {
            if (inverse)
                e = launch_pdl(basis_level_kernel<1, 1>, dim3(g), 256, 0, s, X, pitch, rows, wcols, level);
            else
                e = launch_pdl(basis_level_kernel<1, 0>, dim3(g), 256, 0, s, X, pitch, rows, wcols, level);
        } else {
            if (inverse)
                e = launch_pdl(basis_level_kernel<2, 1>, dim3(g), 256, 0, s, X, pitch, rows, wcols, level);
            else
                e = launch_pdl(basis_level_kernel<2, 0>, dim3(g), 256, 0, s, X, pitch, rows, wcols, level);
        }
        BMM_CUDA_TRY(e);
    }
    return BMM_OK;
}

}  // namespace bmm
