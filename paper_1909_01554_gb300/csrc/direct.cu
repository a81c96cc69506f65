// Small products in one launch: C = A B on the CUDA cores straight from B as
// the caller holds it (m x k times k x n, packed along n), with no transposed
// copy of B, no scratch and no second kernel.
//
// A CTA owns a 64 x 64 tile of C (sizes are multiples of 64: no padding) over
// a slice of k. Per 2048 bits of k, 128 threads each bring 32 rows of one
// 32-bit word of B and transpose the 32 x 32 block in registers (transpose.cu),
// all 256 bring A's rows; then thread (tx, ty) runs LOP3s on rows ty + 16 i and
// columns tx + 16 j (i, j < 4) from shared rows of both operands along k, as
// popc_gemm.cu does. Where the tiles alone leave SMs idle, k is split over the
// CTAs of a cluster, and rank 0 combines their 64 result words (512 bytes)
// through its shared memory.
//
// What bounds it: latency (launch, one round trip to memory, a transpose of
// 256 instructions) up to some 10^8 bit products, the LOP3 rate beyond (a step
// of 2048 bits: 2.1 us of LOP3s a tile and SM, 3.9 measured with two CTAs an
// SM, 4 for one alone). Steps of 1024 and 512 bits, and three or four CTAs an SM
// at 80 or 64 registers, were slower on all but the shortest k.
#include "internal.h"
#include "pdl.cuh"
#include "transpose32.cuh"

namespace bmm {
namespace {

constexpr int TILE = 64;
constexpr int CHUNK_W64 = DIRECT_CHUNK / 64;  // 64-bit words of k per step
constexpr int CHUNK_W32 = 2 * CHUNK_W64;
constexpr int LDW = CHUNK_W32 + 4;         // padded shared row: 16-byte loads of 8 rows on 8 bank groups
constexpr int THREADS = 256;
constexpr int A_ROWS = THREADS / CHUNK_W64, A_LOADS = TILE / A_ROWS;  // rows of A loaded at a time
constexpr int MAX_SPLIT = 8;

__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Rank r of the cluster (blockIdx.z) takes words [r * slice, (r + 1) * slice) of k.
template <int OP, bool SPLIT>
__global__ void __launch_bounds__(THREADS, 2)
    direct_kernel(const uint64_t* A, const uint64_t* B, uint64_t* C, int64_t m, int64_t k, int64_t n, int64_t slice) {
    __shared__ __align__(16) uint32_t sA[TILE * LDW], sB[TILE * LDW];
    __shared__ uint64_t part[MAX_SPLIT][TILE];
    if (SPLIT) cluster_arrive();  // waited for before rank 0's shared memory is written
    wait_for_operands();
    dependents_may_launch();

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tx = tid & 15, ty = tid >> 4;
    const int ar = tid / CHUNK_W64, aw = tid % CHUNK_W64;  // this thread's row and word of A
    const int64_t kw = k / 64, nw = n / 64;
    const int64_t row0 = (int64_t)blockIdx.y * TILE, cw = blockIdx.x;
    const int64_t w0 = SPLIT ? (int64_t)blockIdx.z * slice : 0;
    const int64_t w1 = SPLIT && w0 + slice < kw ? w0 + slice : kw;

    uint32_t acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = 0u;

    for (int64_t at = w0; at < w1; at += CHUNK_W64) {
        const int words = (int)(w1 - at < CHUNK_W64 ? w1 - at : CHUNK_W64);
        // words of 16 bytes that the inner loop runs over: pad with zeros to that
        const int padded = (words + 1) & ~1;
        uint64_t a[A_LOADS];
        const uint64_t* asrc = A + (row0 + ar) * kw + at + aw;
#pragma unroll
        for (int i = 0; i < A_LOADS; i++) a[i] = aw < words ? asrc[i * A_ROWS * kw] : 0ull;
        const int bc = tid & 1, bk = tid >> 1;  // word column, block of 32 rows of B
        uint32_t v[32];
        const bool mine = bk < 2 * padded;
        if (mine) {
            if (bk < 2 * words) {
                const uint32_t* bsrc =
                    reinterpret_cast<const uint32_t*>(B + (at * 64 + 32 * bk) * nw + cw) + bc;
#pragma unroll
                for (int i = 0; i < 32; i++) v[i] = bsrc[2 * i * nw];
            } else {
#pragma unroll
                for (int i = 0; i < 32; i++) v[i] = 0u;
            }
        }
        if (at != w0) __syncthreads();  // the last step's operands have been read
        if (aw < padded) {
#pragma unroll
            for (int i = 0; i < A_LOADS; i++)
                *reinterpret_cast<uint64_t*>(&sA[(ar + i * A_ROWS) * LDW + 2 * aw]) = a[i];
        }
        if (mine) {
            transpose32(v);
#pragma unroll
            for (int i = 0; i < 32; i++) sB[(32 * bc + i) * LDW + bk] = v[i];
        }
        __syncthreads();
#pragma unroll 2
        for (int kk = 0; kk < 2 * padded; kk += 4) {
            uint4 x[4], y[4];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                x[i] = *reinterpret_cast<const uint4*>(&sA[(ty + 16 * i) * LDW + kk]);
                y[i] = *reinterpret_cast<const uint4*>(&sB[(tx + 16 * i) * LDW + kk]);
            }
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    if (OP == OP_GF2) {
                        acc[i][j] ^= x[i].x & y[j].x;
                        acc[i][j] ^= x[i].y & y[j].y;
                        acc[i][j] ^= x[i].z & y[j].z;
                        acc[i][j] ^= x[i].w & y[j].w;
                    } else {
                        acc[i][j] |= x[i].x & y[j].x;
                        acc[i][j] |= x[i].y & y[j].y;
                        acc[i][j] |= x[i].z & y[j].z;
                        acc[i][j] |= x[i].w & y[j].w;
                    }
                }
        }
    }

    // Row 2 warp + half + 16 i of the tile (half = lane / 16): ballots of its
    // four groups of 16 columns; lane 2 i + half keeps the word.
    uint64_t word = 0;
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const bool bit = OP == OP_GF2 ? (__popc(acc[i][j]) & 1) != 0 : acc[i][j] != 0u;
            const uint32_t bal = __ballot_sync(0xffffffffu, bit);
            if (lane == 2 * i) word |= (uint64_t)(bal & 0xffffu) << (16 * j);
            if (lane == 2 * i + 1) word |= (uint64_t)(bal >> 16) << (16 * j);
        }
    const int row = 2 * warp + (lane & 1) + 16 * (lane >> 1);
    if (!SPLIT) {
        if (lane < 8) C[(row0 + row) * nw + cw] = word;
        return;
    }
    cluster_wait();  // every CTA of the cluster runs
    if (lane < 8) {
        uint32_t dst;
        asm("mapa.shared::cluster.u32 %0, %1, 0;"
            : "=r"(dst)
            : "r"((uint32_t)__cvta_generic_to_shared(&part[blockIdx.z][row])));
        asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(dst), "l"(word) : "memory");
    }
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    if (blockIdx.z == 0 && tid < TILE) {
        uint64_t w = part[0][tid];
        for (unsigned z = 1; z < gridDim.z; z++) w = OP == OP_GF2 ? w ^ part[z][tid] : w | part[z][tid];
        C[(row0 + tid) * nw + cw] = w;
    }
}

}  // namespace

cudaError_t launch_direct(int op, const uint64_t* A, const uint64_t* B, uint64_t* C, int64_t m,
                          int64_t k, int64_t n, int split, cudaStream_t s) {
    const int64_t kw = k / 64, slice = (kw + split - 1) / split;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = 1;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = (unsigned)split;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n / 64), (unsigned)(m / 64), (unsigned)split);
    cfg.blockDim = dim3(THREADS);
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = split > 1 ? 2 : 1;
    TraceScope ts(BMM_PHASE_BASE, s);
    if (split > 1)
        return op == OP_GF2 ? cudaLaunchKernelEx(&cfg, direct_kernel<OP_GF2, true>, A, B, C, m, k, n, slice)
                            : cudaLaunchKernelEx(&cfg, direct_kernel<OP_BOOL, true>, A, B, C, m, k, n, slice);
    return op == OP_GF2 ? cudaLaunchKernelEx(&cfg, direct_kernel<OP_GF2, false>, A, B, C, m, k, n, slice)
                        : cudaLaunchKernelEx(&cfg, direct_kernel<OP_BOOL, false>, A, B, C, m, k, n, slice);
}

}  // namespace bmm
