// FP64 complex GEMMs on the tcgen05 tensor cores by exact integer slicing
// (the Ozaki scheme): the large FP64 products of the plan update, the FP64
// fit and its adjoint, and the exchange application.
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"
#include "oz_sizes.cuh"
#include "zgemm.cuh"

// Plan-owned scratch for the slices and the row scales.
struct OzWork {
    __half *sa, *sb;                 // slices of the A rows and of the rotated B rows
    size_t cap_a, cap_b;             // capacity in halves
    int *ma, *mb;                    // row exponents and row-maximum parts of the operands
    size_t cap_ma, cap_mb;           // capacity in ints
    int *gsum;                       // exact int32 group sums
    size_t cap_g;                    // capacity in ints: a whole product's (oz_gsum_ints) or a chunk's (oz_chunk_ints)
    long long wait_budget;           // cycle budget of the pipeline waits (0: the default; < 0: test hook)
};

// Ints of group sums of a whole product, and of the rows that keep every CTA pair busy for two tiles.
size_t oz_gsum_ints(int M, int N, int batch);
size_t oz_chunk_ints(int M, int N);

// True if g (single or batched, complex128 or complex64 operands, complex128 output) can
// run with the given scratch.
bool oz_fits(const ZGemm &g, const OzWork &w);

// C = alpha op(A) op(B) + beta C with the ZGemm conventions (strides, conj,
// lower_only, kmode, k_to_m_end, batch); the result carries an error of the
// order of an FP64 GEMM's (slices of 8 bits, 56 bits per operand, products of
// slice pairs with s + t <= 8). Device errors go to *err: 1 for a bounded wait
// that gave up, 2 for an infinite or NaN operand entry (first error wins).
isdf_status oz_zgemm(const ZGemm &g, const OzWork &w, int *err, cudaStream_t st);
