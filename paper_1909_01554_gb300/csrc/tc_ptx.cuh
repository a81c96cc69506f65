// PTX wrappers shared by the tensor-core kernels: mbarriers with bounded
// waits, TMA loads, tcgen05 MMAs, commits and TMEM access, and the expansion
// of packed bits and the packing of result bits in registers.
#pragma once

#include "tile_order.h"
#include <cuda.h>
#include <stdint.h>

#include "internal.h"
#include "tc_batched.h"

namespace bmm {
namespace {

constexpr int BN = TC_TILE_N;    // columns of C per tile (UMMA N)
constexpr int TMEM_COLS = 512;

constexpr uint64_t WAIT_NS = 2000000000ull;  // 2 s

// ---------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint64_t globaltimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_arrive_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase of `bar` with the given parity. Returns false
// (after recording the timeout) if it did not complete within WAIT_NS.
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, uint32_t* err,
                                            uint64_t limit_ns = WAIT_NS) {
    const uint64_t t0 = globaltimer();
    for (uint32_t i = 1;; i++) {
        if (mbar_try(bar, parity)) return true;
        if ((i & 255u) == 0 && globaltimer() - t0 > limit_ns) {
            atomicOr(err, DEVERR_TIMEOUT);
            return false;
        }
    }
}

// Arrive on the barrier at the same shared-memory offset in CTA `cta` of
// the cluster. What the waiter goes on to use is this CTA's own shared
// memory and TMEM, read by the pair's tensor cores; the writer orders it
// with fence.proxy.async.shared::cta or tcgen05.fence before arriving, so a
// CTA-scope arrive is enough (a cluster-scope release costs a memory barrier).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar, uint32_t cta) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(bar), "r"(cta));
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// Every thread of both CTAs of the cluster (no thread may have exited).
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void fence_barrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t* err) {
    if (mbar_try(bar, parity)) return true;
    return mbar_wait_slow(bar, parity, err);
}

__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y,
                                            int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

// Shared-memory matrix descriptor for a K-major operand in the 128-byte
// swizzled canonical layout: each row's 128 bytes of k sit at row * 128,
// 8-row groups form 1024-byte atoms (SBO = 1024 between them), and within an
// atom the 16-byte chunk c of row r is stored at chunk c ^ (r % 8). The
// start address may point k bytes into the first row (k < 128): the swizzle
// is applied to absolute address bits, so atoms must be 1024-byte aligned.
// Adding 2 to the descriptor advances the start address by 32 bytes.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;              // LBO: unused for swizzled K-major, 1 by convention
    d |= (uint64_t)(1024u >> 4) << 32;   // SBO: 8-row atom stride
    d |= (uint64_t)1 << 46;              // descriptor version for tcgen05
    d |= (uint64_t)2 << 61;              // layout: 128-byte swizzle
    return d;
}

// Instruction descriptor for kind::f8f6f4: D format (1 = F32), A and B
// format 0 (E4M3), both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
template <int M, int N = BN>
__host__ __device__ constexpr uint32_t instr_desc(uint32_t dfmt) {
    return (dfmt << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Instruction descriptor for kind::mxf4 (block-scaled e2m1, FP32
// accumulate): A and B format 1 (E2M1) at bits 7 and 10, both K-major,
// N >> 3 at bit 17, scale format 1 (UE8M0) at bit 23, M >> 4 at bit 24;
// scale-factor data ids 0 and K = 64 (bit 31 clear).
template <int M, int N = BN>
__host__ __device__ constexpr uint32_t instr_desc_mxf4() {
    return (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | (1u << 23) |
           ((uint32_t)(M >> 4) << 24);
}

// D (TMEM) += A (TMEM) x B (shared, descriptor). PAIR: cta_group::2, issued
// by the even CTA of the pair; A, B and D are the two CTAs' halves at the
// same TMEM / shared-memory addresses.
template <bool PAIR>
__device__ __forceinline__ void mma_f8_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t db,
                                          uint32_t idesc, uint32_t accumulate) {
    if (PAIR)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
            "r"(tmem_a), "l"(db), "r"(idesc), "r"(accumulate)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
            "r"(tmem_a), "l"(db), "r"(idesc), "r"(accumulate)
            : "memory");
}

// As mma_f8_ta for e2m1 operands with block scales: every 32 k of a row of
// A (B) is scaled by the UE8M0 byte the tensor core reads from TMEM at
// tmem_sfa (tmem_sfb); here every scale byte holds the same value.
template <bool PAIR>
__device__ __forceinline__ void mma_f4_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t db,
                                          uint32_t idesc, uint32_t tmem_sfa, uint32_t tmem_sfb,
                                          uint32_t accumulate) {
    if (PAIR)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %6, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X"
            " [%0], [%1], %2, %3, [%4], [%5], p;\n\t}" ::"r"(tmem_d),
            "r"(tmem_a), "l"(db), "r"(idesc), "r"(tmem_sfa), "r"(tmem_sfb), "r"(accumulate)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %6, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X"
            " [%0], [%1], %2, %3, [%4], [%5], p;\n\t}" ::"r"(tmem_d),
            "r"(tmem_a), "l"(db), "r"(idesc), "r"(tmem_sfa), "r"(tmem_sfb), "r"(accumulate)
            : "memory");
}

// Arrive on `bar` once every MMA this thread issued so far has completed.
// PAIR: on the barrier at the same offset in each CTA of `mask`.
template <bool PAIR>
__device__ __forceinline__ void mma_commit(uint32_t bar, uint16_t mask = 3) {
    if (PAIR)
        asm volatile(
            "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
            " [%0], %1;" ::"r"(bar),
            "h"(mask)
            : "memory");
    else
        asm volatile(
            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
            : "memory");
}

template <bool PAIR>
__device__ __forceinline__ void tmem_alloc(uint32_t slot) {
    if (PAIR) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
}

template <bool PAIR>
__device__ __forceinline__ void tmem_dealloc(uint32_t tmem) {
    if (PAIR)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(TMEM_COLS)
                     : "memory");
    else
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(TMEM_COLS)
                     : "memory");
}

// 32 lanes x 64 columns (one row per thread), then wait for the load.
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, uint32_t (&v)[64]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, "
        "%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, "
        "%48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, "
        "[%64];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
          "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]),
          "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]),
          "=r"(v[31]), "=r"(v[32]), "=r"(v[33]), "=r"(v[34]), "=r"(v[35]), "=r"(v[36]),
          "=r"(v[37]), "=r"(v[38]), "=r"(v[39]), "=r"(v[40]), "=r"(v[41]), "=r"(v[42]),
          "=r"(v[43]), "=r"(v[44]), "=r"(v[45]), "=r"(v[46]), "=r"(v[47]), "=r"(v[48]),
          "=r"(v[49]), "=r"(v[50]), "=r"(v[51]), "=r"(v[52]), "=r"(v[53]), "=r"(v[54]),
          "=r"(v[55]), "=r"(v[56]), "=r"(v[57]), "=r"(v[58]), "=r"(v[59]), "=r"(v[60]),
          "=r"(v[61]), "=r"(v[62]), "=r"(v[63])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 32 lanes x 64 columns: one row per thread, 64 consecutive 32-bit columns
// (both operand stages of a packed stage in one instruction; TMEM stores
// share the tensor pipe's issue path with the MMAs, so fewer, wider ones).
__device__ __forceinline__ void tmem_st64(uint32_t taddr, const uint32_t (&v)[64]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x64.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32, "
        "%33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, %48, "
        "%49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63, %64};" ::"r"(
            taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
        "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]),
        "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]),
        "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]),
        "r"(v[29]), "r"(v[30]), "r"(v[31]), "r"(v[32]), "r"(v[33]), "r"(v[34]), "r"(v[35]),
        "r"(v[36]), "r"(v[37]), "r"(v[38]), "r"(v[39]), "r"(v[40]), "r"(v[41]), "r"(v[42]),
        "r"(v[43]), "r"(v[44]), "r"(v[45]), "r"(v[46]), "r"(v[47]), "r"(v[48]), "r"(v[49]),
        "r"(v[50]), "r"(v[51]), "r"(v[52]), "r"(v[53]), "r"(v[54]), "r"(v[55]), "r"(v[56]),
        "r"(v[57]), "r"(v[58]), "r"(v[59]), "r"(v[60]), "r"(v[61]), "r"(v[62]), "r"(v[63])
        : "memory");
}

// ---------------------------------------------------------------- expansion
// Packed word x holds 32 consecutive k of one row. Output word j (j = 0..7)
// gets bit (8t + j) of x in byte t, moved to bit 3 of that byte (e4m3 0x08 =
// 2^-6). The moves are multiplications by powers of two (left) or high
// halves of them (right) with factors the compiler cannot see, so they run
// on the FMA pipe and leave the integer pipe the masks alone.
struct Spread {
    uint32_t f[8];  // f[j]: 2^(3-j) for j <= 3 (low product), 2^(35-j) for j > 3 (high)
    uint32_t g[4];  // spread4: 2, 1 (low products), 2^31, 2^30 (high)
};

__device__ __forceinline__ void spread8(uint32_t x, const Spread& sp, uint32_t* y) {
    constexpr uint32_t mask = 0x08080808u;
    y[0] = (x * sp.f[0]) & mask;
    y[1] = (x * sp.f[1]) & mask;
    y[2] = (x * sp.f[2]) & mask;
    y[3] = x & mask;
    y[4] = __umulhi(x, sp.f[4]) & mask;
    y[5] = __umulhi(x, sp.f[5]) & mask;
    y[6] = __umulhi(x, sp.f[6]) & mask;
    y[7] = __umulhi(x, sp.f[7]) & mask;
}

// e2m1 form: output word j (j = 0..3) gets bit (4t + j) of x in nibble t,
// moved to bit 1 of the nibble (e2m1 0x2 = 1.0, scaled by 2^-6 at the MMA,
// so products are 2^-12 as in the e4m3 form).
__device__ __forceinline__ void spread4(uint32_t x, const Spread& sp, uint32_t* y) {
    constexpr uint32_t mask = 0x22222222u;
    y[0] = (x * sp.g[0]) & mask;
    y[1] = x & mask;
    y[2] = __umulhi(x, sp.g[2]) & mask;
    y[3] = __umulhi(x, sp.g[3]) & mask;
}

// UE8M0 block scale 2^-6 (biased exponent 121) in every byte.
constexpr uint32_t SCALE_WORD = 0x79797979u;

// 32 result bits of one accumulator row slice -> one word, bit j from v[j].
// GF(2): v[j] = count * 2^-12 exactly; adding 2^11 puts count's LSB in bit 0.
// Boolean: any non-zero count. Each bit goes in with one funnel shift (the
// word shifts right by one and takes the bit at the top), in four
// independent chains of eight that are merged at the end.
template <int OP>
__device__ __forceinline__ uint32_t pack_bits(const uint32_t* v) {
    uint32_t c[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int j = 0; j < 8; j++)
#pragma unroll
        for (int g = 0; g < 4; g++) {
            const uint32_t x = v[8 * g + j];
            const uint32_t bit = OP == OP_GF2 ? __float_as_uint(__uint_as_float(x) + 2048.0f)
                                              : min(x, 1u);  // fp32 counts are >= 0
            c[g] = __funnelshift_r(c[g], bit, 1);  // bit 0 of `bit` enters at bit 31
        }
    // chain g holds bits 8g..8g+7 in its top byte
    return (c[0] >> 24) | (c[1] >> 16) | (c[2] >> 8) | c[3];
}

// As TileOrder::tile.
__device__ __forceinline__ TileCoord tile_of(int t, int tiles_m, int tiles_n) {
    const int per_leaf = tiles_m * tiles_n;
    TileCoord c;
    c.leaf = t / per_leaf;
    int r = t - c.leaf * per_leaf;
    const int group = GROUP_M * tiles_n;
    const int g = r / group;
    const int first_m = g * GROUP_M;
    const int gm = min(GROUP_M, tiles_m - first_m);
    const int in = r - g * group;
    c.tm = first_m + in % gm;
    c.tn = in / gm;
    return c;
}

// 16 bytes global -> shared, asynchronous (cp.async; wait with cp_async_wait_all).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}

__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap* m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}

}  // namespace
}  // namespace bmm
