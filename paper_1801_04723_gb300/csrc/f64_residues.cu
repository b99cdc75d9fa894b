// Large FP64 products on the BF16 tensor cores, by residues (crt.cu).
//
// GB300's FP64 pipe does 1.25 TFLOP/s; 18 or 19 exact BF16 products of signed
// 8-bit residues give the same 2 m n k at 60 to 90 TFLOP/s, with operands in
// 63-bit fixed point relative to the largest entry of their row (column) and
// the sum itself exact.  Whether that is as accurate as 53-bit floating point
// depends on the entries: an entry is off by at most 2^-63 of its row's (or
// column's) largest, so the residue form's error is at most
//     2^-63 (S_i + T_j) rowmax_i colmax_j,   S_i = sum_k |a_ik| / rowmax_i,
// T_j alike, the FP64 kernel's k 2^-53 G_ij with G_ij = sum_k |a_ik| |b_kj|.
// The first is the smaller one wherever k G_ij >= 2^-10 (S_i + T_j) rowmax_i
// colmax_j.  A lower bound of G_ij for every output comes from the sizes of the
// entries alone: sorted by size, the g-th eighth of a row (g = 1 .. 7) is at
// least 2^-(s_g + 1) of the row's largest, s_g from its exponents, and the worst
// a column can do is to pair its eighths in the opposite order (the
// rearrangement inequality), so
//     G_ij >= (k / 8) sum_{g=1..6} 2^-(s_g + 1) 2^-(t_{7-g} + 1) rowmax_i colmax_j
// and
//     k^2 sum_{g=1..6} 2^-(s_g + t_{7-g}) >= 2^-5 (S + T)
// is enough for every output.  The exponents pass finds the largest s_g and
// t_g of the operands and bounds S and T, a one-thread kernel compares, and
// either the residue product or the FP64 kernel runs (the other one's launches
// return at once): operands with an infinity or NaN, mostly empty ones and
// widely spread ones keep the FP64 kernel, without a host read.  A Gram matrix
// and its inverse pass by 5 bits and more; a strictly diagonally dominant one
// (entries U(-1, 1) beside a diagonal n, its inverse's diagonal 4 n times the
// entries beside it) by 2 at n = 8192 and k = 4096, at k = 512 it does not
// (S + T = 2 k, which any operands have, would pass one bit less: order 8192
// took 60.2 ms that way, and 36.3 this way).
#include "crt.h"
#include "f64_residues.h"
#include "split.h"

namespace spin {
namespace {

constexpr int kMinBits = 63;
constexpr size_t kHeader = 256;  // spread[2 * kSpreadInts], use[2] (residues, FP64 kernel)
constexpr int kUse = 2 * kSpreadInts;

__global__ void choose_form_kernel(const int* spread, double k, int* use) {
    double sum = 0.0;
    for (int g = 1; g < kSpreadLevels; g++)
        sum += ldexp(1.0, -min(spread[g - 1] + spread[kSpreadInts + 6 - g], 1000));
    const double mass = ldexp((double)spread[kSpreadLevels] + (double)spread[kSpreadInts + kSpreadLevels], -14);
    const int residues = k * k * sum >= 0.03125 * mass;
    use[0] = residues;
    use[1] = !residues;
}

size_t exps_bytes(int64_t m, int64_t n) { return ((size_t)(m + n) * sizeof(int) + 255) / 256 * 256; }

}  // namespace

int f64_residue_moduli(int64_t k) {
    const CrtFormat f = crt_format(k, kMinBits);
    return f.moduli;  // 0 where the moduli do not give the 63 bits of the rule above
}

size_t f64_residue_bytes(int64_t m, int64_t n, int64_t k, bool least) {
    const int mods = f64_residue_moduli(k);
    if (mods == 0) return 0;
    return kHeader + 256 + exps_bytes(m, n) + (least ? crt_min_bytes(m, n, k, mods) : crt_full_bytes(m, n, k, mods));
}

int f64_residue_decide(const F64Product& p, void* arena, F64Plan* plan, cudaStream_t s) {
    unsigned char* base = (unsigned char*)(((uintptr_t)arena + 255) & ~(uintptr_t)255);
    int* head = (int*)base;
    plan->use_residues = head + kUse;
    plan->use_fp64 = head + kUse + 1;
    plan->ea = (int*)(base + kHeader);
    plan->eb = plan->ea + p.m;
    plan->rest = base + kHeader + exps_bytes(p.m, p.n);
    SPIN_CUDA_TRY(cudaMemsetAsync(head, 0, 2 * kSpreadInts * sizeof(int), s));
    SplitSource src;
    src.A = p.A;
    src.lda = p.lda;
    src.B = p.B;
    src.ldb = p.ldb;
    const int rc = launch_exponents(src, (int)p.m, (int)p.n, (int)p.k, plan->ea, plan->eb, nullptr, nullptr, head, s);
    if (rc) return rc;
    choose_form_kernel<<<1, 1, 0, s>>>(head, (double)p.k, head + kUse);
    SPIN_CUDA_TRY(cudaGetLastError());
    return SPIN_OK;
}

int f64_residue_product(const F64Product& p, const F64Plan& plan, size_t arena_bytes, const void* arena, int* err,
                        cudaStream_t s) {
    CrtProduct q = {};
    q.m = p.m;
    q.n = p.n;
    q.k = p.k;
    q.min_bits = kMinBits;
    q.alpha = p.alpha;
    q.beta = p.beta;
    q.A = p.A;
    q.lda = p.lda;
    q.B = p.B;
    q.ldb = p.ldb;
    q.C = p.C;
    q.ldc = p.ldc;
    q.D = p.D;
    q.ldd = p.ldd;
    q.active = plan.use_residues;
    q.a_exps = plan.ea;
    q.b_exps = plan.eb;
    q.err = err;
    const size_t used = (size_t)((const unsigned char*)plan.rest - (const unsigned char*)arena);
    return crt_product(q, plan.rest, arena_bytes - used, s);
}

}  // namespace spin
