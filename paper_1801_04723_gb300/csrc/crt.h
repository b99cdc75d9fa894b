// Exact integer products on the BF16 tensor cores by residues (crt.cu).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "tc_gemm.h"

namespace spin {

constexpr int kCrtMinModuli = 8;  // 31 bits at k = 1
constexpr int kCrtMaxModuli = 19;  // 63 bits at k = 98304
constexpr int kCrtMaxBits = 63;  // signed in 64 bits
constexpr int kCrtFewBits = 55;  // up to here 96-bit fractions and four pieces do (crt.cu, split.cu)

// Pairwise coprime, in falling order; signed residues |r| <= 128.
__host__ __device__ constexpr int crt_modulus(int l) {
    constexpr int p[kCrtMaxModuli] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227,
                                      223, 217, 211, 199, 197, 193, 191, 181, 179};
    return p[l];
}

// Moduli and fixed-point bits per operand for an inner dimension k: the
// fewest moduli whose product exceeds twice the largest |sum| at bits >=
// min_bits, then every bit that they allow (at most kCrtFewBits for a min_bits
// up to it, kCrtMaxBits above).  0 moduli: none fits.
struct CrtFormat {
    int moduli;
    int bits;
};
CrtFormat crt_format(int64_t k, int min_bits);

// Bits that stand in for s 8-bit digit slices (pairs t + u < s): the digits'
// own, so the operands are the same fixed-point integers and nothing is left
// out of their product: for every operand the residue form's error is the
// digit form's less that of the pairs it leaves out.  Fewer bits would be
// worse for operands whose rows are full of entries near the largest (four
// bits fewer, one modulus fewer: 4.8 times the digit form's error for normal
// entries at k = 128, where the operands' rounding is all of it).
inline int crt_bits_for_slices(int s) { return 8 * s - 1; }

// One operand's or the whole product's device memory.
//   exps       one int per row of A / column of B, for all of them
//   planes     [panel of rows] x moduli BF16 planes, K-major
//   residues   moduli bytes per output of a panel pair
// crt_min_bytes: the least arena that crt_product accepts; crt_full_bytes:
// the arena that holds everything in one panel pair (count problems).
size_t crt_full_bytes(int64_t m, int64_t n, int64_t k, int moduli, int count = 1);
size_t crt_min_bytes(int64_t m, int64_t n, int64_t k, int moduli, int count = 1);

// D = beta*C + alpha*(A B) (+ I), alpha = +-1, beta = 0 or 1, for `count`
// problems (count = 0: one problem given by plain pointers).  Views, sums of squares, active flags
// and statuses as in TcGemmParams.
struct CrtProduct {
    int64_t m, n, k;
    int min_bits;
    double alpha, beta;
    int add_identity;
    // one problem
    const double* A;
    int64_t lda;
    const double* B;
    int64_t ldb;
    const double* C;
    int64_t ldc;
    double* D;
    int64_t ldd;
    // count problems
    int count;
    BatchView Av, Bv, Cv, Dv;
    const int* active;    // optional, device
    const int* valid;     // optional, device: sums of squares cover the leading valid[z] x valid[z] block
    double* sumsq_a;      // optional, device: += sum of squares of A (one entry per problem)
    double* sumsq_b;
    double* sumsq_d;
    const int* a_exps;    // optional, device: row exponents of A from an earlier product with the same A
    const int* b_exps;    // optional, device (with a_exps): column exponents of B, n per problem
    int* a_exps_out;      // optional, device: m ints per problem, where they are kept (else in the arena)
    int* err;
};
// Launches, all on s; *launches (optional) counts them.
int crt_product(const CrtProduct& p, void* arena, size_t bytes, cudaStream_t s, int* launches = nullptr);

}  // namespace spin
