// Sizes of the exact-slicing products (ozaki.cu) that the scratch of a plan is planned from: plain C++, no CUDA.
#pragma once

#include <stddef.h>
#include <stdint.h>

constexpr int OTK = 64;       // K chunk (halves)
constexpr int OTM = 128;      // rows of A and of Bh loaded by each CTA of a pair
constexpr int NSLICE = 7;
constexpr int KSLAB = 7168;   // complex K of one pass: 9 2^14 14,336 < 2^31
constexpr int PK = 256;       // complex k of one row-maximum part

constexpr int64_t oz_round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// complex K of one pass over the operands: all of it up to KSLAB, else equal slabs (multiples of 32)
constexpr int oz_slab(int K)
{
    const int n = (K + KSLAB - 1) / KSLAB;
    return n <= 1 ? K : (int)oz_round_up((K + n - 1) / n, 32);
}

// Halves of slices and ints of exponents that hold an M x N product (batch products) of K terms or of any smaller
// number: equal slabs do not grow with K (65,536 has slabs of 6,560, 42,464 of 7,104), so room is made for the longest
// slab up to K.
inline void oz_sizes(int M, int N, int K, int batch, size_t *halves_a, size_t *halves_b, size_t *ints_a, size_t *ints_b)
{
    const int slab = K < KSLAB ? K : KSLAB;
    const int64_t Ra = oz_round_up(M, OTM), Rb = oz_round_up(2 * (int64_t)N, OTM), Kp = oz_round_up(2 * (int64_t)slab, OTK);
    const size_t parts = (size_t)((slab + PK - 1) / PK);
    *halves_a = (size_t)batch * NSLICE * Ra * Kp;
    *halves_b = (size_t)batch * NSLICE * Rb * Kp;
    *ints_a = (size_t)batch * M * (1 + parts);
    *ints_b = (size_t)batch * N * (1 + parts);
}
