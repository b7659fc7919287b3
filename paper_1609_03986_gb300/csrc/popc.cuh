// Population count of a 512-bit XOR (a Hamming distance) split between the logic
// pipe and the population-count pipe (shared by the brute-force and the dense
// CUDA-core matchers).
#pragma once

#include <stdint.h>

namespace latch {

// carry-save adder: a + b + c = 2 h + l, bit by bit
__device__ __forceinline__ void csa(uint32_t& h, uint32_t& l, uint32_t a, uint32_t b, uint32_t c) {
    const uint32_t u = a ^ b;
    h = (a & b) | (u & c);
    l = u ^ c;
}

// half adder: a + b = 2 h + l
__device__ __forceinline__ void hadd(uint32_t& h, uint32_t& l, uint32_t a, uint32_t b) {
    h = a & b;
    l = a ^ b;
}

// Hamming weight of 16 words.  Words 0-10 go through a carry-save adder tree that folds
// them into one word each of weight 1, 2, 4 and 8 (7 adders and a half adder, 16 logic
// operations; 4 population counts for 11), words 11-15 through a population count each:
// 9 counts and 32 logic operations with the XORs.  Folding 8 words takes 12 counts and 30
// operations and held the population-count pipe (16 lanes per clock against 64) fullest.
// Measured (GB300, 8 / 9 / 11 words folded): 10,000 x 10,000 on the CUDA cores 339 / 315 /
// 306 us, 16,384 x 131,072 6,558 / 6,064 / 5,885 us, the dense matcher at 640x480 and
// radius 8 255 / 246 / 248 us (as it was written then; 238 now).
__device__ __forceinline__ int popc16(const uint32_t (&x)[16]) {
    uint32_t h0, h1, h2, h3, h4, l0, l1, l2, l3, ones;
    csa(h0, l0, x[0], x[1], x[2]);
    csa(h1, l1, x[3], x[4], x[5]);
    csa(h2, l2, x[6], x[7], x[8]);
    csa(h3, l3, l0, l1, l2);
    csa(h4, ones, l3, x[9], x[10]);
    uint32_t f0, t0, f1, twos, eights, fours;
    csa(f0, t0, h0, h1, h2);     // weight 2: t0, h3, h4; weight 4: f0
    csa(f1, twos, t0, h3, h4);   // weight 4: f0, f1
    hadd(eights, fours, f0, f1);
    const int tree = 8 * __popc(eights) + 4 * __popc(fours) + 2 * __popc(twos) + __popc(ones);
    return tree + (__popc(x[11]) + __popc(x[12])) + (__popc(x[13]) + __popc(x[14])) + __popc(x[15]);
}

}  // namespace latch
