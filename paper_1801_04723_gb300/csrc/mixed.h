// Mixed-precision level products (mixed.cu).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "tc_gemm.h"

namespace spin {

// What the FP64-class products are as accurate as, in 8-bit digit slices.
constexpr int kSchurSlices = 7;  // Schur complements (55 bits)
constexpr int kLevelSlices = 4;  // level products in SPIN_MIXED_DIGITS (31 bits)
constexpr int kMaxResidualSlices = 7;

// Digit slices of the refinement residual R = I - A X.  The error of the
// computed rel = ||R||_F / (||A||_F ||X||_F) is modelled as
// residual_error_model(n, s); a residual that certifies a result (a
// stopping decision) keeps it within 1 % of tol, the first residual, which
// only feeds the Newton-Schulz update (its error enters the next residual
// additively), within 20 %; each decision adds the model error of its own
// residual to rel before comparing with tol.
double residual_error_model(int64_t n, int s);
int residual_slices_for(int64_t n, double tol);
int first_residual_slices_for(int64_t n, double tol, int sr);
// Products smaller than this in m or n stay in FP64: below it a product has
// a handful of 128 x 256 tiles and a short K, so the tensor-core path (two
// operand splits and a launch that fills a few SMs) costs more than the FP64
// kernel, whose small tiles fill the SMs.  Measured single inversions, bf16x3
// to 1e-10: threshold 128 -> 384 took n = 512 / 1024 / 2048 / 4096 from
// 3.29 / 6.10 / 13.1 / 30.0 ms to 1.82 / 4.57 / 10.4 / 24.7 ms (512 gives the
// same times; 384 keeps orders like 777 on the tensor cores).
constexpr int64_t kTcMin = 384;

// Slice-pair schedules of the tensor-core product forms (fill pa, pb, pg,
// num_pairs and the exactness fields of p).
void tc_pairs_bf16x3(TcGemmParams& p);           // planes hi, lo: hi hi + hi lo + lo hi
void tc_pairs_bf16x6(TcGemmParams& p);           // planes hi, mid, lo: pairs of weight >= 2^-16
void tc_pairs_ozaki(TcGemmParams& p, int slices);  // digit pairs t + u < slices, exact runs of 1024

// A growable device arena for split planes.
struct MixScratch {
    void* base = nullptr;
    size_t cap = 0;
    size_t refused_at = 0;
    int reserve(size_t need, size_t want);  // at least need bytes, want where the device has them
};

size_t bf16x3_scratch_bytes(int64_t m, int64_t n, int64_t k);
size_t bf16x6_scratch_bytes(int64_t m, int64_t n, int64_t k);
size_t ozaki_scratch_bytes(int64_t m, int64_t n, int64_t k, int slices);

int gemm_bf16x3(int64_t m, int64_t n, int64_t k, double alpha, const double* A, int64_t lda, const double* B,
                int64_t ldb, double beta, const double* C, int64_t ldc, double* D, int64_t ldd, void* scratch,
                size_t scratch_bytes, int* err, cudaStream_t s);

// FP64-class product (the Schur complements, the refinement residual, the
// level products of SPIN_MIXED_DIGITS): as accurate as s digit slices, by
// residues (crt.cu) for s >= 4, else by digits (s <= 3, and k beyond 96 runs of
// 1024).  At n = 2048 the residues take as many tensor-core products for s = 4
// (10), 12 instead of 15, 14 instead of 21 and 16 instead of 28 for s = 7, and
// their drain is cheaper: us by digits and by residues, s = 4 to 7: 425, 528,
// 656, 784 and 227, 256, 279, 307; n = 512: 107, 124, 140, 157 and 30, 30, 31, 35.
int fp64_class_moduli(int64_t k, int slices);       // 0: digits
size_t fp64_class_least(int64_t m, int64_t n, int64_t k, int slices);  // the least arena
size_t fp64_class_bytes(int64_t m, int64_t n, int64_t k, int slices);  // an arena that needs no panels
double fp64_class_products(int64_t k, int slices);  // tensor-core products of m x n x k
// The residue form runs in panels in any arena of at least the digit form's
// size (from order 40 on); library-owned arenas are made larger, up to this, to save the panels'
// repeated splits and launches at small orders.
constexpr size_t kFp64ClassArena = (size_t)2 << 30;
struct Fp64ClassExtra {
    const int* active = nullptr;  // optional, device int: runs only while nonzero
    double* sumsq_a = nullptr;    // optional, device: += sums of squares of A, B and D
    double* sumsq_b = nullptr;
    double* sumsq_d = nullptr;
    int* a_exps = nullptr;        // optional, device: m row exponents of A, kept between products
    bool digits = false;          // by digits for every s: the arena may be too small for the residues
    bool a_known = false;         // a_exps and *sumsq_a are there from an earlier product with this A
};
int gemm_fp64_class(int64_t m, int64_t n, int64_t k, double alpha, const double* A, int64_t lda, const double* B,
                    int64_t ldb, double beta, const double* C, int64_t ldc, double* D, int64_t ldd, int slices,
                    int add_identity, const Fp64ClassExtra& x, void* scratch, size_t scratch_bytes, int* err,
                    cudaStream_t s);

// Split-then-multiply in two halves so callers can time them separately.
struct SplitPlan {
    uint16_t* a;    // A planes (rows of A, K-major)
    uint16_t* b;    // B planes (columns of B as rows, K-major)
    int* ea;        // ozaki: row exponents of A
    int* eb;        // ozaki: column exponents of B
    int64_t ld;
    int slices;     // ozaki slice count (bf16x3: 2 planes)
};
int plan_bf16x3(int64_t m, int64_t n, int64_t k, void* scratch, size_t bytes, SplitPlan* sp);
int plan_ozaki(int64_t m, int64_t n, int64_t k, int slices, void* scratch, size_t bytes, SplitPlan* sp);
// Both operands' BF16 planes (2 or 3, the plan's) in one launch.
// active (optional, device int): the split / product runs only while *active != 0.
int split_bf16(const SplitPlan& sp, const double* A, int64_t lda, const double* B, int64_t ldb, int64_t m, int64_t n,
               int64_t k, cudaStream_t s, const int* active = nullptr);
int product_bf16x3(const SplitPlan& sp, int64_t m, int64_t n, int64_t k, double alpha, double beta, const double* C,
                   int64_t ldc, double* D, int64_t ldd, int* err, cudaStream_t s);
// Three-plane form (hi, mid, lo) with the six products of weight <= 2^-16.
int plan_bf16x6(int64_t m, int64_t n, int64_t k, void* scratch, size_t bytes, SplitPlan* sp);
int product_bf16x6(const SplitPlan& sp, int64_t m, int64_t n, int64_t k, double alpha, double beta, const double* C,
                   int64_t ldc, double* D, int64_t ldd, int* err, cudaStream_t s, const int* active = nullptr);
int product_ozaki(const SplitPlan& sp, int64_t m, int64_t n, int64_t k, double alpha, double beta, const double* C,
                  int64_t ldc, double* D, int64_t ldd, int add_identity, double* sumsq, int* err, cudaStream_t s,
                  const int* active = nullptr);

// Device-side Newton-Schulz control (refine.cu) for `count` matrices whose
// info records (INFO_WORDS int32 each) start at `records`:
//   init    active[z] = (status of z == 0), rel[z] = -1, iters[z] = 0;
//   decide  for every active z: rel[z] = sqrt(nR[z]) / (sqrt(nA[z]) sqrt(nX[z])),
//           iters[z] = it, nX[z] = nR[z] = 0 for the next round; off when rel <= tol, or (recording
//           SPIN_ERR_NOT_CONVERGED) when rel is not finite or it >= max_refine;
//   finish  a nonzero *err (a bounded wait that gave up) becomes the status of
//           every matrix still at SPIN_OK.
int launch_refine_init(const int32_t* records, int count, int* active, double* rel, int* iters, cudaStream_t s);
// margin: the model error of this round's residual; converged when rel + margin <= tol.
int launch_refine_decide(const double* nA, double* nX, double* nR, int count, double tol, double margin,
                         int it, int max_refine, int* active, double* rel, int* iters, int32_t* records,
                         cudaStream_t s);
int launch_refine_finish(const int* err, int32_t* records, int count, cudaStream_t s);

}  // namespace spin
