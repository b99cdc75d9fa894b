// Operand splits of the tensor-core products (split.cu): row and column
// exponents, and BF16 planes of both operands, one launch each.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace spin {

// The operands of one product, or of `count` products (count > 0: device
// views): A (m x k, rows of A become the planes' rows) and B (k x n, columns
// of B become the planes' rows).
struct SplitSource {
    int count = 0;
    const double* A = nullptr;
    int64_t lda = 0;
    const double* B = nullptr;
    int64_t ldb = 0;
    BatchView Av{}, Bv{};
    const int* active = nullptr;  // optional, device: problem z only while active[z] != 0 (count = 0: active[0])
    const int* valid = nullptr;   // optional, device: sums of squares of problem z cover its leading valid[z] block
};

// Exponents e with |a_ik| < 2^e for every row i of A (k entries) and every
// column j of B: ea (m per problem, or null: not wanted), eb (n per problem,
// or null), += sums of squares (optional, one entry per problem).  spread
// (optional, device int[2 * kSpreadInts], count = 0 only): entry g - 1 of A's
// half is raised to the largest over the rows (of B's half: over the columns)
// of the least t of 0 .. 25 such that 8 - g eighths of the row's exponents are
// at least its largest - t; 1000 where none is or an entry is not finite; the
// last entry to the largest bound of a row's sum of sizes over its largest
// size, in units of 2^-14.  Rows of zeros do not count.
constexpr int kSpreadLevels = 7, kSpreadInts = kSpreadLevels + 1;
int launch_exponents(const SplitSource& src, int m, int n, int k, int* ea, int* eb, double* sumsq_a, double* sumsq_b,
                     int* spread, cudaStream_t s);

// What a plane holds.
enum SplitKind {
    SPLIT_BF16,      // planes 2 or 3: hi, (mid,) lo of the value in FP32
    SPLIT_DIGITS,    // planes 1..7: balanced base-256 digits relative to the row's exponent
    SPLIT_RESIDUES,  // planes: residues of the value in `bits` fixed-point bits (crt.h)
};
// Rows row0 .. row0 + rows - 1 of A and columns col0 .. col0 + cols - 1 of B
// (rows or cols 0: not that operand), to planes of rows x k (cols x k)
// entries, leading dimension ld (a multiple of 8), problem after problem:
// dst + (z * planes + q) * rows * ld.  ea, eb: m (n) exponents per problem.
struct SplitTarget {
    SplitKind kind;
    int planes, bits;
    int m, n, k;
    int row0, rows, col0, cols;
    const int* ea;
    const int* eb;
    uint16_t* a;
    uint16_t* b;
    int64_t ld;
};
int launch_split(const SplitSource& src, const SplitTarget& t, cudaStream_t s);

}  // namespace spin
