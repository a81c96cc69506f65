// Planner and executor for one product (the accelerator-side layers of
// Sec. 3.4 on a single GPU with all operands resident in HBM):
//   transpose B -> Bt (Sec. 3.5), then `serial` depth-first levels
//   (Sec. 3.8: combine, recurse, fold, reusing scratch across the 7
//   branches), then `depth - serial` breadth-first levels merged into one
//   expanding pass over both operands (Sec. 3.9, 3.15), the batched base case over
//   the 7^d leaves (Sec. 3.10), and one compressing pass (Sec. 3.11).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "plan.h"
#include "slp.h"
#include "tc_batched.h"

namespace bmm {

cudaError_t launch_expand(int variant, int d, const uint64_t* A, int64_t lda, int64_t m,
                          uint32_t amask, uint64_t* TL, const uint64_t* B, int64_t ldb, int64_t n,
                          uint32_t bmask, uint64_t* SL, int64_t kw, cudaStream_t s);
cudaError_t launch_compress(int variant, int d, const uint64_t* leaves, int64_t lr, int64_t lw,
                            uint64_t* C, int64_t ldc, uint32_t dest, uint32_t first,
                            cudaStream_t s);
cudaError_t launch_combine(int operand, const uint64_t* X, int64_t pitch, int64_t hr, int64_t hw,
                           uint32_t mask, uint64_t* dst, cudaStream_t s);
cudaError_t launch_fold(const uint64_t* R, int64_t hr, int64_t hw, uint64_t* C, int64_t ldc,
                        uint32_t dest, uint32_t first, cudaStream_t s);
bmm_status run_tc_strided(int op, int path, const uint64_t* A, int64_t lda, int64_t strideA,
                          const uint64_t* Bt, int64_t ldb, int64_t strideB, uint64_t* C,
                          int64_t ldc, int64_t strideC, int64_t count, int64_t m, int64_t k,
                          int64_t n, cudaStream_t s);

namespace {

constexpr uint64_t ALIGN = 256;
uint64_t round_up(uint64_t x) { return (x + ALIGN - 1) / ALIGN * ALIGN; }

constexpr int MAX_MERGED = 2;  // breadth-first levels merged in registers

int ipow7(int d) {
    int r = 1;
    while (d-- > 0) r *= 7;
    return r;
}

bool divisible(int64_t m, int64_t k, int64_t n, int d) {
    const int64_t unit = (int64_t)64 << d;
    return (m % ((int64_t)1 << d) == 0) && (m >> d) % 64 == 0 && k % unit == 0 && n % unit == 0;
}

// The last depth-first level hands its branches straight to the
// breadth-first passes: its input combination is done by the expanding pass
// (reading the parent's quadrants) and its output fold by the compressing
// pass, so that level needs no branch buffers.
bool fused_last_serial(int depth, int serial) { return serial > 0 && depth > serial; }

// Bytes of scratch for a plan: Bt, the depth-first branch buffers of every
// serial level, and the breadth-first leaves at the bottom.
uint64_t workspace_for(int64_t m, int64_t k, int64_t n, int depth, int serial) {
    uint64_t b = round_up((uint64_t)k * n / 8);  // Bt
    const int bufs = fused_last_serial(depth, serial) ? serial - 1 : serial;
    for (int l = 1; l <= bufs; l++) {
        b += round_up((uint64_t)(m >> l) * (k >> l) / 8);
        b += round_up((uint64_t)(n >> l) * (k >> l) / 8);
        b += round_up((uint64_t)(m >> l) * (n >> l) / 8);
    }
    const int dp = depth - serial;
    if (dp > 0) {
        const uint64_t r = (uint64_t)ipow7(dp);
        b += round_up(r * (uint64_t)(m >> depth) * (k >> depth) / 8);
        b += round_up(r * (uint64_t)(n >> depth) * (k >> depth) / 8);
        b += round_up(r * (uint64_t)(m >> depth) * (n >> depth) / 8);
    }
    return b;
}

struct Exec {
    const Plan& p;
    const int od;  // levels outside the base case (the last one may run inside it)
    char* ws;
    cudaStream_t s;
    uint32_t xi[7], eta[7], zeta[4];
    uint64_t* Bt = nullptr;
    uint64_t* Apad = nullptr;  // A with k padded to kp (only when kp != k)
    uint64_t* T[8] = {nullptr};
    uint64_t* S[8] = {nullptr};
    uint64_t* R[8] = {nullptr};
    uint64_t *TL = nullptr, *SL = nullptr, *QL = nullptr;

    Exec(const Plan& plan, void* w, cudaStream_t st)
        : p(plan), od(plan.depth - plan.kernel_level), ws((char*)w), s(st) {
        switch (p.variant) {
            case 0: slp::level_masks<0>(xi, eta, zeta); break;
            case 1: slp::level_masks<1>(xi, eta, zeta); break;
            default: slp::level_masks<2>(xi, eta, zeta); break;
        }
        uint64_t off = 0;
        auto take = [&](uint64_t bytes) {
            uint64_t* q = (uint64_t*)(ws + off);
            off += round_up(bytes);
            return q;
        };
        Bt = take((uint64_t)p.kp * p.n / 8);
        if (p.kp != p.k) Apad = take((uint64_t)p.m * p.kp / 8);
        const int bufs = fused_last_serial(od, p.serial) ? p.serial - 1 : p.serial;
        for (int l = 1; l <= bufs; l++) {
            T[l] = take((uint64_t)(p.m >> l) * (p.kp >> l) / 8);
            S[l] = take((uint64_t)(p.n >> l) * (p.kp >> l) / 8);
            R[l] = take((uint64_t)(p.m >> l) * (p.n >> l) / 8);
        }
        const int dp = od - p.serial;
        if (dp > 0) {
            const uint64_t r = (uint64_t)ipow7(dp);
            TL = take(r * (uint64_t)(p.m >> od) * (p.kp >> od) / 8);
            SL = take(r * (uint64_t)(p.n >> od) * (p.kp >> od) / 8);
            QL = take(r * (uint64_t)(p.m >> od) * (p.n >> od) / 8);
        }
    }

    // The product of `count` blocks below the outer levels (strides in words):
    // the base case, or the innermost Strassen level with the base case
    // inside one kernel.
    bmm_status blocks(const uint64_t* A, int64_t lda, int64_t sa, const uint64_t* B, int64_t ldb,
                      int64_t sb, uint64_t* C, int64_t ldc, int64_t sc, int64_t count, int64_t m,
                      int64_t k, int64_t n) {
        if (p.kernel_level) {
            LevelMasks lm;
            std::memcpy(lm.xi, xi, sizeof xi);
            std::memcpy(lm.eta, eta, sizeof eta);
            std::memcpy(lm.zeta, zeta, sizeof zeta);
            if (p.path == BMM_PATH_TC_FP4_PAIR)
                return run_tc_level(A, lda, sa, B, ldb, sb, C, ldc, sc, count, m, k, n, lm, s);
            BMM_CUDA_TRY(launch_popc_level(A, lda, sa, B, ldb, sb, C, ldc, sc, count, m, k, n, lm,
                                           s));
            return BMM_OK;
        }
        return run_base_product_batched(p.op, p.path, A, lda, sa, B, ldb, sb, C, ldc, sc, count,
                                        m, k, n, s);
    }

    bmm_status level(int l, const uint64_t* A, int64_t lda, const uint64_t* B, int64_t ldb,
                     uint64_t* C, int64_t ldc, int64_t m, int64_t k, int64_t n) {
        if (l < p.serial) {
            const int64_t hm = m / 2, hk = k / 2, hn = n / 2;
            uint32_t first = 0xF;
            if (l + 1 == p.serial && fused_last_serial(od, p.serial)) {
                for (int h = 0; h < 7; h++) {
                    uint32_t dest = 0;
                    for (int q = 0; q < 4; q++) dest |= ((zeta[q] >> h) & 1u) << q;
                    if (!dest) continue;
                    bmm_status st = leaves(A, lda, xi[h], B, ldb, eta[h], C, ldc, dest,
                                           first & dest, hm, hk, hn);
                    if (st != BMM_OK) return st;
                    first &= ~dest;
                }
                return BMM_OK;
            }
            for (int h = 0; h < 7; h++) {
                BMM_CUDA_TRY(launch_combine(0, A, lda, hm, hk / 64, xi[h], T[l + 1], s));
                BMM_CUDA_TRY(launch_combine(1, B, ldb, hn, hk / 64, eta[h], S[l + 1], s));
                bmm_status st = level(l + 1, T[l + 1], hk / 64, S[l + 1], hk / 64, R[l + 1],
                                      hn / 64, hm, hk, hn);
                if (st != BMM_OK) return st;
                uint32_t dest = 0;
                for (int q = 0; q < 4; q++) dest |= ((zeta[q] >> h) & 1u) << q;
                if (dest) {
                    BMM_CUDA_TRY(launch_fold(R[l + 1], hm, hn / 64, C, ldc, dest, first & dest, s));
                    first &= ~dest;
                }
            }
            return BMM_OK;
        }
        if (od == l) return blocks(A, lda, 0, B, ldb, 0, C, ldc, 0, 1, m, k, n);
        return leaves(A, lda, 0, B, ldb, 0, C, ldc, 0, 0, m, k, n);
    }

    // The breadth-first levels below an m x k x n block: expand both operands
    // into the leaves, the batched base case, compress into C. With non-zero
    // masks the block's operands are combinations of the quadrants of A / B
    // (their parents) and the result is folded into the quadrants `dest` of
    // C (its parent), as a depth-first level would.
    bmm_status leaves(const uint64_t* A, int64_t lda, uint32_t amask, const uint64_t* B,
                      int64_t ldb, uint32_t bmask, uint64_t* C, int64_t ldc, uint32_t dest,
                      uint32_t first, int64_t m, int64_t k, int64_t n) {
        const int dp = od - p.serial;
        const int64_t lm = m >> dp, lk = k >> dp, ln = n >> dp;
        BMM_CUDA_TRY(launch_expand(p.variant, dp, A, lda, m, amask, TL, B, ldb, n, bmask, SL, k / 64, s));
        const int64_t count = ipow7(dp);
        bmm_status st = blocks(TL, lk / 64, lm * lk / 64, SL, lk / 64, ln * lk / 64, QL, ln / 64,
                               lm * ln / 64, count, lm, lk, ln);
        if (st != BMM_OK) return st;
        BMM_CUDA_TRY(launch_compress(p.variant, dp, QL, lm, ln / 64, C, ldc, dest, first, s));
        return BMM_OK;
    }
};

}  // namespace

// Scratch of a plan with k padded to kp (the padded copy of A when kp != k).
uint64_t workspace_padded(int64_t m, int64_t k, int64_t kp, int64_t n, int depth, int serial) {
    return workspace_for(m, kp, n, depth, serial) + (kp != k ? round_up((uint64_t)m * kp / 8) : 0);
}

// Both sides' time in us, fitted to measurements of each inside a graph. Direct: a
// CTA's step of 2048 bits of k takes 1.1 us + 2.8 us of work when the SMs are
// shared, 4 us alone after 2 us of launch and epilogue (3 us with a cluster).
// Tensor: 6.3 us for the two launches, 0.27 us per 384 bits of k and round of
// tiles, 0.8 us between rounds, 0.5 us per MB of transposed B, 0.5 us where tiles
// are sliced. Over 60 shapes of 10^5 to 10^10 bit products the choice is within 9 %
// of the better side, 0.5 % on average. Measured (direct / tensor): 64^3 2.1 / 5.7,
// 256 x 512 x 384 2.9 / 6.7, 1024^3 6.6 / 7.8, 64 x 4096 x 64 3.5 / 6.2, 2496 x 1088 x
// 384 6.7 / 8.0; past the line, 128 x 8192 x 2048 10.0 / 9.3, 64 x 32768 x 64 9.7 /
// 6.7, 1024 x 256 x 4096 10.1 / 6.8, 2048 x 512 x 1600 10.8 / 7.5.
int direct_split_for(int64_t m, int64_t k, int64_t n) {
    if (m / 64 > 65535 || m / 64 * (n / 64) > 65535) return 0;
    const double sms = sm_count();
    const double tiles = (double)(m / 64) * (double)(n / 64);
    const double rounds = std::ceil(std::ceil(m / 256.0) * std::ceil(n / 256.0) / (sms / 2));
    const int slice = rounds > 1 ? 0 : tc_fp4_slice_stages(m, k, n, nullptr);
    double best = 6.3 + rounds * 0.27 * (slice ? slice : std::ceil(k / 384.0)) + (rounds - 1) * 0.8 +
                  0.5e-6 * ((double)k * n / 8) + (slice ? 0.5 : 0.0);
    int split = 0;
    for (int s = 1; s <= 8; s *= 2) {
        const double bits = std::ceil(k / 64.0 / s) * 64.0;
        const double steps = std::ceil(bits / DIRECT_CHUNK), work = bits / DIRECT_CHUNK;
        double per_sm = tiles * s / sms;
        if (per_sm <= 2) per_sm = std::ceil(per_sm);
        const double alone = (s > 1 ? 3.0 : 2.0) + 4.0 * work;
        const double shared = 1.5 + per_sm * (1.1 * steps + 2.8 * work);
        const double t = std::max(alone, shared);
        if (t < best) {
            best = t;
            split = s;
        }
    }
    return split;
}

bmm_status make_plan(int op, int64_t m, int64_t k, int64_t n, const bmm_opts* opts, Plan* out,
                     bool ask_memory) {
    bmm_opts o;
    bmm_opts_default(&o);
    if (opts) o = *opts;
    Plan p;
    p.op = op;
    p.m = m;
    p.k = k;
    p.n = n;
    if (o.variant < 0 || o.variant > 2) return BMM_ERR_INVALID;
    if (o.kernel_level < 0 || o.kernel_level > 1) return BMM_ERR_INVALID;
    p.variant = o.variant;
    if (o.path < BMM_PATH_AUTO || o.path > BMM_PATH_TC_FP4_PAIR) return BMM_ERR_INVALID;
    if (is_tc_path(o.path) && !tc_path_available()) return BMM_ERR_UNSUPPORTED;
    if (o.path == BMM_PATH_TC_FP4_PAIR && !tc_fp4_available()) return BMM_ERR_UNSUPPORTED;
    // recursion depth
    if (op == OP_BOOL) {
        if (o.strassen_depth > 0) return BMM_ERR_INVALID;  // no additive inverse
        p.depth = 0;
    } else if (o.strassen_depth >= 0) {
        p.depth = o.strassen_depth;
        if (p.depth > 6) return BMM_ERR_UNSUPPORTED;
        if (p.depth > 0 && !divisible(m, k, n, p.depth)) return BMM_ERR_UNSUPPORTED;
    } else {
        // Auto: recurse while every leaf dimension stays >= 8192 (below that the
        // base case loses efficiency faster than 7/8 of the work is saved).
        int d = 0;
        while (d < 4 && divisible(m, k, n, d + 1) && (m >> (d + 1)) >= 8192 &&
               (k >> (d + 1)) >= 8192 && (n >> (d + 1)) >= 8192)
            d++;
        p.depth = d;
    }
    // A tuned choice (bmm_autotune) replaces the rules below when both the
    // path and the depth are left to the library.
    const bool path_left = o.path == BMM_PATH_AUTO;
    int tpath = 0, tdepth = 0;
    const bool tuned = o.path == BMM_PATH_AUTO && o.strassen_depth < 0 && o.kernel_level == 0 &&
                       tuned_choice(op, m, k, n, &tpath, &tdepth) &&
                       (tdepth == 0 || (op == OP_GF2 && divisible(m, k, n, tdepth)));
    if (tuned) {
        p.depth = tdepth;
        o.path = tpath;
    }
    // base-case path (auto_path below); the tensor paths pad k so that every
    // leaf's k is a multiple of 128 bits
    p.path = o.path == BMM_PATH_AUTO ? auto_path() : o.path;
    // The innermost level inside the base-case kernel: the CUDA-core kernel
    // and the e2m1 SM-pair kernel have that form; a plan without Strassen
    // levels has no level to move.
    p.kernel_level = (o.kernel_level && p.depth > 0) ? 1 : 0;
    if (p.kernel_level && p.path != BMM_PATH_POPC && p.path != BMM_PATH_TC_FP4_PAIR)
        return BMM_ERR_UNSUPPORTED;
    p.kp = k;
    if (is_tc_path(p.path)) {
        // leaf k a multiple of 128 bits; with the level in the tensor kernel,
        // of its 512-bit packed stage (a quadrant's copies stay inside it)
        const int64_t unit = (int64_t)(p.kernel_level ? 512 : 128) << p.depth;
        p.kp = (k + unit - 1) / unit * unit;
    }
    const int od = p.depth - p.kernel_level;  // levels run by the XOR passes
    // depth-first levels: at least od - MAX_MERGED; more while the
    // breadth-first scratch does not fit in free device memory.
    int serial_min = od > MAX_MERGED ? od - MAX_MERGED : 0;
    if (o.serial_depth >= 0) {
        if (o.serial_depth > od) return BMM_ERR_INVALID;
        p.serial = o.serial_depth < serial_min ? serial_min : o.serial_depth;
    } else {
        p.serial = serial_min;
        size_t fr = 0, tot = 0;
        if (ask_memory && p.serial < od && !o.workspace &&
            cudaMemGetInfo(&fr, &tot) == cudaSuccess) {
            fr += scratch_idle_bytes();
            while (p.serial < od &&
                   workspace_padded(m, k, p.kp, n, od, p.serial) > (uint64_t)(fr * 0.9))
                p.serial++;
        }
    }
    p.workspace_bytes = workspace_padded(m, k, p.kp, n, od, p.serial);
    // (a record of the e2m1 path at depth 0 was timed in this form)
    if (path_left && p.path == BMM_PATH_TC_FP4_PAIR && p.depth == 0)
        p.direct_split = direct_split_for(m, k, n);
    *out = p;
    return BMM_OK;
}

uint64_t plan_pass_bytes(const Plan& p) {
    uint32_t xi[7], eta[7], zeta[4];
    switch (p.variant) {
        case 0: slp::level_masks<0>(xi, eta, zeta); break;
        case 1: slp::level_masks<1>(xi, eta, zeta); break;
        default: slp::level_masks<2>(xi, eta, zeta); break;
    }
    auto bits = [](uint32_t x) { return (uint64_t)__builtin_popcount(x); };
    const int d = p.depth - p.kernel_level, dp = d - p.serial;
    const bool fused = fused_last_serial(d, p.serial);
    const uint64_t r = (uint64_t)ipow7(dp > 0 ? dp : 0);
    const uint64_t la = (uint64_t)(p.m >> d) * (p.kp >> d) / 8;
    const uint64_t lb = (uint64_t)(p.n >> d) * (p.kp >> d) / 8;
    const uint64_t lc = (uint64_t)(p.m >> d) * (p.n >> d) / 8;
    // transpose: B read, Bt written with its padding columns
    uint64_t total = (uint64_t)p.k * p.n / 8 + (uint64_t)p.kp * p.n / 8;
    if (p.kp != p.k) total += (uint64_t)p.m * p.k / 8 + (uint64_t)p.m * p.kp / 8;  // padded A
    uint64_t reps = 1;                              // executions of the current level
    for (int l = 0; l < p.serial; l++, reps *= 7) {
        const uint64_t a = (uint64_t)(p.m >> (l + 1)) * (p.kp >> (l + 1)) / 8;
        const uint64_t b = (uint64_t)(p.n >> (l + 1)) * (p.kp >> (l + 1)) / 8;
        const uint64_t c = (uint64_t)(p.m >> (l + 1)) * (p.n >> (l + 1)) / 8;
        const bool last_fused = fused && l + 1 == p.serial;
        uint64_t per = 0;
        uint32_t first = 0xF;
        for (int h = 0; h < 7; h++) {
            uint32_t dest = 0;
            for (int q = 0; q < 4; q++) dest |= ((zeta[q] >> h) & 1u) << q;
            if (last_fused) {  // expand reads the parent's quadrants, compress folds
                if (!dest) continue;
                per += bits(xi[h]) * a + r * la + bits(eta[h]) * b + r * lb;
                per += r * lc + bits(dest) * c + bits(dest & ~first) * c;
            } else {  // combine into branch buffers, fold the branch result
                per += (bits(xi[h]) + 1) * a + (bits(eta[h]) + 1) * b;
                if (dest) per += c + bits(dest) * c + bits(dest & ~first) * c;
            }
            first &= ~dest;
        }
        total += reps * per;
    }
    if (dp > 0 && !fused) {
        const int s = p.serial;
        const uint64_t in_a = (uint64_t)(p.m >> s) * (p.kp >> s) / 8;
        const uint64_t in_b = (uint64_t)(p.n >> s) * (p.kp >> s) / 8;
        const uint64_t out_c = (uint64_t)(p.m >> s) * (p.n >> s) / 8;
        total += reps * (in_a + r * la + in_b + r * lb + r * lc + out_c);
    }
    return total;
}

bmm_status run_cubic_fp4(int op, const uint64_t* A, const uint64_t* B, uint64_t* C, int64_t m,
                         int64_t k, int64_t n, uint64_t* Bt, uint64_t* Apad, cudaStream_t s) {
    const int64_t kw = k / 64, kpw = (kw + 1) / 2 * 2;
    const TransposeJob bt = {B, Bt, n / 64, kpw, k, n, 0};
    const TransposeJob pad = {A, Apad, kw, kpw, m, 0, 1};
    const uint64_t* Aop = kpw != kw ? Apad : A;
    ZeroJob zero = {C, n / 64, m, n, {}};
    const int slice = tc_fp4_slice_stages(m, kpw * 64, n, &zero.tiles);
    BMM_CUDA_TRY(launch_prepare(bt, kpw != kw ? &pad : nullptr, zero, s));
    if (slice)
        return run_fp4_strided(op, Aop, kpw, 0, Bt, kpw, 0, C, n / 64, 0, 1, m, kpw * 64, n, s, slice);
    return run_base_product(op, BMM_PATH_TC_FP4_PAIR, Aop, kpw, Bt, kpw, C, n / 64, m, kpw * 64, n, s);
}

bmm_status execute_plan(const Plan& p, const uint64_t* A, const uint64_t* B, uint64_t* C,
                        void* workspace, cudaStream_t s) {
    if (p.direct_split) {
        BMM_CUDA_TRY(launch_direct(p.op, A, B, C, p.m, p.k, p.n, p.direct_split, s));
        return BMM_OK;
    }
    Exec ex(p, workspace, s);
    if (p.depth == 0 && p.path == BMM_PATH_TC_FP4_PAIR)
        return run_cubic_fp4(p.op, A, B, C, p.m, p.k, p.n, ex.Bt, ex.Apad, s);
    // zero columns k..kp of A (a pitched copy) and of B^T
    const bool padded = p.kp != p.k;
    const TransposeJob bt = {B, ex.Bt, p.n / 64, p.kp / 64, p.k, p.n, 0};
    const TransposeJob pad = {A, ex.Apad, p.k / 64, p.kp / 64, p.m, 0, 1};
    BMM_CUDA_TRY(launch_prepare(bt, padded ? &pad : nullptr, {}, s));
    const uint64_t* Aop = padded ? ex.Apad : A;
    return ex.level(0, Aop, p.kp / 64, ex.Bt, p.kp / 64, C, p.n / 64, p.m, p.kp, p.n);
}

// Base case for BMM_PATH_AUTO: the tensor cores wherever the device has
// them; on SM pairs where clusters can be launched (faster at every measured
// size from 4096^3 up), with e2m1 operands (twice the e4m3 rate from 8192^3
// up); else the CUDA-core kernel.
int auto_path() {
    if (!tc_path_available()) return BMM_PATH_POPC;
    if (tc_fp4_available()) return BMM_PATH_TC_FP4_PAIR;
    return tc_pair_available() ? BMM_PATH_TC_FP8_PAIR : BMM_PATH_TC_FP8;
}

bmm_status run_base_product(int op, int path, const uint64_t* A, int64_t lda, const uint64_t* Bt,
                            int64_t ldb, uint64_t* C, int64_t ldc, int64_t m, int64_t k,
                            int64_t n, cudaStream_t s) {
    return run_base_product_batched(op, path, A, lda, 0, Bt, ldb, 0, C, ldc, 0, 1, m, k, n, s);
}

bmm_status run_base_product_batched(int op, int path, const uint64_t* A, int64_t lda,
                                    int64_t strideA, const uint64_t* Bt, int64_t ldb,
                                    int64_t strideB, uint64_t* C, int64_t ldc, int64_t strideC,
                                    int64_t count, int64_t m, int64_t k, int64_t n,
                                    cudaStream_t s) {
    if (count <= 0) return BMM_OK;
    if (path == BMM_PATH_POPC) {
        BMM_CUDA_TRY(launch_popc_nt(op, A, lda, strideA, Bt, ldb, strideB, C, ldc, strideC, count,
                                    m, k, n, s));
        return BMM_OK;
    }
    return run_tc_strided(op, path, A, lda, strideA, Bt, ldb, strideB, C, ldc, strideC, count, m,
                          k, n, s);
}

}  // namespace bmm
