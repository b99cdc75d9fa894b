// Large FP64 products by residues on the tensor cores (f64_residues.cu).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "common.cuh"

namespace spin {

// Inversions whose top products are all larger than this have an arena, i.e.
// orders above 4096.  A 2048^3 product takes 14 ms on the FP64 pipe and 0.6 ms
// by residues, so the line is not where the residues stop paying; it lies there
// because orders up to 4096 are held to the FP64 kernel elsewhere:
// spin_model_seconds prices it (within 25 % of the measured inversion at n =
// 4096), and up to 1024 the batched, the persistent and the no-allocation
// forms, which have no residue arena, give the single inversion's bits.
constexpr int64_t kF64ResidueTop = 2048;
// In those inversions products whose m, n and k are all above this take the
// residue form.  Time per product, FP64 kernel and residues: 1024^3 1.75 and
// 0.15 ms, 512^3 0.27 and 0.053, 256^3 0.061 and 0.045 (level sums on two
// streams).  Whole inversions with the line at 2048, 1000, 500, 250 and 120:
// order 8192 259.5, 48.3, 38.3, 38.4 and 43.5 ms, 5000 69.5, 26.8, 18.1, 17.1
// and 19.0 ms, 4161 41.2, 29.4, 14.0, 12.8 and 15.1 ms.
constexpr int64_t kF64ResidueMin = 256;
// Most device memory of one product's arena: a 16384^3 product then runs in
// panels (its planes and residues take 24 GB at once).
constexpr size_t kF64ResidueArena = (size_t)8 << 30;

struct F64Product {
    int64_t m, n, k;
    double alpha, beta;
    const double* A;
    int64_t lda;
    const double* B;
    int64_t ldb;
    const double* C;
    int64_t ldc;
    double* D;
    int64_t ldd;
};
struct F64Plan {
    const int* use_residues;  // device flags, one of them set
    const int* use_fp64;
    int *ea, *eb;
    void* rest;
};
int f64_residue_moduli(int64_t k);  // 0: no such form for this k
// Arena of one product: the least, or the one that needs no panels.
size_t f64_residue_bytes(int64_t m, int64_t n, int64_t k, bool least);
// Exponents, and which form runs; then the residue product (a no-op on the
// device when the FP64 kernel, gated by use_fp64, is to run).
int f64_residue_decide(const F64Product& p, void* arena, F64Plan* plan, cudaStream_t s);
int f64_residue_product(const F64Product& p, const F64Plan& plan, size_t arena_bytes, const void* arena, int* err,
                        cudaStream_t s);

}  // namespace spin
