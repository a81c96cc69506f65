// The bit transpose of a 32 x 32 block in one thread's registers.
#pragma once

#include <stdint.h>

namespace bmm {

// v[i] = row i of a 32 x 32 bit block; afterwards v[i] = its column i.
__device__ __forceinline__ void transpose32(uint32_t (&v)[32]) {
#pragma unroll
    for (int i = 0; i < 16; i++) {
        const uint32_t a = v[i], b = v[i + 16];
        v[i] = __byte_perm(a, b, 0x5410);
        v[i + 16] = __byte_perm(a, b, 0x7632);
    }
#pragma unroll
    for (int i = 0; i < 32; i++) {
        if (i & 8) continue;
        const uint32_t a = v[i], b = v[i + 8];
        v[i] = __byte_perm(a, b, 0x6240);
        v[i + 8] = __byte_perm(a, b, 0x7351);
    }
#pragma unroll
    for (int j = 4; j > 0; j >>= 1) {
        const uint32_t mask = j == 4 ? 0x0F0F0F0Fu : j == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
        for (int i = 0; i < 32; i++) {
            if (i & j) continue;
            const uint32_t a = v[i], b = v[i + j];
            v[i] = (a & mask) | ((b << j) & ~mask);
            v[i + j] = ((a >> j) & mask) | (b & ~mask);
        }
    }
}

}  // namespace bmm
