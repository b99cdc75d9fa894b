// Operand splits of the tensor-core products.
//
// Both operands of a product in one launch: the products of a recursion at
// small orders are bound by launches, and two half-empty launches cost more
// than one.  A thread block takes a tile of one operand:
//   A   32 rows x 128 columns, a warp per row, 4 consecutive columns per lane;
//   B   128 rows x 32 columns, transposed through shared memory, a warp per
//       column, 4 consecutive rows per lane;
// so that every plane is written in 8-byte pieces, 256 bytes per warp.  Bound
// by HBM (8 bytes read, 2 written per plane and entry) for the BF16 and digit
// planes, by FP32 arithmetic (6 operations per residue) for the residues.  A
// warp's rows (columns) are a loop that is not unrolled: the residues' code is
// long, and four copies of it per side came from memory on every launch (both
// operands of 512^2 to 15 moduli: 29 -> 12 us; of 2048^2 73 -> 63; to 16 moduli 11
// and 61).
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "crt.h"
#include "split.h"

namespace spin {
namespace {

// ------------------------------------------------------------- sources --

struct SideOne {
    const double* p;
    int64_t ld;
    __device__ __forceinline__ const double* row(int, int r) const { return p + (int64_t)r * ld; }
};
struct SideMany {
    BatchView v;
    __device__ __forceinline__ const double* row(int z, int r) const {
        const int64_t l = v.ld_of(z);
        return v.base[z] + (v.r0 + r) * l + v.c0;
    }
};

__device__ __forceinline__ bool problem_on(const int* active, int z) { return active == nullptr || active[z] != 0; }

// ----------------------------------------------------------- exponents --

// Biased exponent field of x (0 for zero and subnormals).  The exponent e
// with max|x| < 2^e (frexp convention) of a row is max(field) - 1022: the
// largest magnitude has the largest field.  Integer work only.
__device__ __forceinline__ int exp_field(double x) {
    return (int)((unsigned long long)__double_as_longlong(x) >> 52) & 0x7FF;
}

constexpr int kSpreadSteps = 26;  // t = 0, 1, ..., 25
constexpr int kNoSpread = 1000;

// The spread counts: per thread 32 bins of 16 bits in shared memory, bin d the
// entries whose exponent is d below the largest (31: further, or 0), two bins a
// word and a bank per lane, so that one shared add per entry is all (26
// comparisons and additions in registers took 3/4 of the pass's time; a thread
// sees at most 98304 / 16 entries).
constexpr int kSpreadWords = 16;
__device__ __forceinline__ void count_entry(unsigned (*bins)[32], int lane, double v, int top) {
    const int f = exp_field(v), d = f == 0 ? 31 : min(top - f, 31);
    atomicAdd(&bins[d >> 1][lane], 1u << ((d & 1) * 16));
}
// One bin after the other, from 0: the least t of 0 .. 25 with at least
// (8 - g) / 8 k entries in bins 0 .. t, and an upper bound of the sum of the
// entries' sizes over the largest, in units of 2^-14 (an entry of bin d is
// below 2^(1 - d) of the largest; every other one counts a unit).
struct SpreadScan {
    int seen = 0, t = kNoSpread, mass = 0;
    __device__ __forceinline__ void next(int i, int count, int k, int g) {
        seen += count;
        mass += count * max(16384 >> max(i - 1, 0), 1);
        if (t == kNoSpread && 8ll * seen >= (long long)(8 - g) * k) t = i;
    }
    // entry g of the result: a level, or behind them the sum
    __device__ __forceinline__ int result(int k, int g, int top) const {
        if (g > kSpreadLevels) return mass + (k - seen);
        return top == 0x7FF ? kNoSpread : t;  // an infinity or NaN
    }
};
__device__ __forceinline__ bool not_zero(double v) {
    return ((unsigned)__double2hiint(v) << 1 | (unsigned)__double2loint(v)) != 0u;  // no FP64 operation
}

constexpr int kExpWarps = 16;
// Loads a thread has in flight: one warp walks a row (16 warps a block of 32
// columns), so few warps share an SM and latency bounds the pass.  Both
// operands of 2048^2: 18.8 us, 36.6 with one load of A and four of B at a time
// and one form of the kernel for everything; of 4096^2 50.7 and 87 us (268 MB:
// 40 us).
constexpr int kExpLoads = 8;
// A load that stays before the next one: left to itself the compiler takes
// them one by one and waits for each.
__device__ __forceinline__ double load_now(const double* p) {
    double v;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}

// Blocks [0, blocks_a): kExpWarps rows of A, a warp each; the others: 32
// columns of B, all warps over the rows.  SPREAD: the counts of the large FP64
// products' rule too; SUM: sums of squares (sumsq_a, sumsq_b, each may be
// null).  Forms of their own: under a run-time condition the compiler computes
// the squares for everyone and selects afterwards, on the FP64 pipe, and the
// counts take 32 KB of shared memory.
template <class Side, bool SPREAD, bool SUM>
__global__ void __launch_bounds__(32 * kExpWarps)
exponents_kernel(Side A, Side B, int m, int n, int k, int blocks_a, int* __restrict__ ea, int* __restrict__ eb,
                 double* sumsq_a, double* sumsq_b, int64_t sss, int* spread, const int* active, const int* valid) {
    const int z = blockIdx.y;
    if (!problem_on(active, z)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nv = valid ? valid[z] : 0x7fffffff;
    __shared__ int smax[kExpWarps][32];
    __shared__ int scount[SPREAD ? 32 : 1][kSpreadSteps + 1];  // the last one: the column has a nonzero entry
    __shared__ unsigned bins[SPREAD ? kExpWarps : 1][kSpreadWords][32];
    static_assert(kSpreadSteps % 2 == 0 && kSpreadSteps / 2 <= kExpWarps && kSpreadSteps < 2 * kSpreadWords, "bins");
    __shared__ double ssum[kExpWarps];
    double ss = 0.0;
    double* sum;
    if ((int)blockIdx.x < blocks_a) {
        sum = sumsq_a;
        const int r = (int)blockIdx.x * kExpWarps + warp;
        if (r < m) {
            const double* p = A.row(z, r);
            const bool sum_row = sum != nullptr && r < nv;
            int top = 0;
            int c = lane;
            for (; c + 32 * (kExpLoads - 1) < k; c += 32 * kExpLoads) {
                double v[kExpLoads];
#pragma unroll
                for (int u = 0; u < kExpLoads; u++) v[u] = load_now(p + c + 32 * u);
#pragma unroll
                for (int u = 0; u < kExpLoads; u++) {
                    top = max(top, exp_field(v[u]));
                    if (SUM && sum_row && c + 32 * u < nv) ss = fma(v[u], v[u], ss);
                }
            }
            for (; c < k; c += 32) {
                const double v = p[c];
                top = max(top, exp_field(v));
                if (SUM && sum_row && c < nv) ss = fma(v, v, ss);
            }
            top = __reduce_max_sync(0xffffffffu, top);
            if (lane == 0) ea[(int64_t)z * m + r] = top - 1022;
            if constexpr (SPREAD) {
#pragma unroll
                for (int j = 0; j < kSpreadWords; j++) bins[warp][j][lane] = 0u;
                bool nonzero = top != 0;
                if (!nonzero)  // zeros and subnormals
                    for (int c = lane; c < k; c += 32) nonzero |= not_zero(p[c]);
                int c = lane;
                for (; c + 32 * (kExpLoads - 1) < k; c += 32 * kExpLoads) {
                    double v[kExpLoads];
#pragma unroll
                    for (int u = 0; u < kExpLoads; u++) v[u] = load_now(p + c + 32 * u);
#pragma unroll
                    for (int u = 0; u < kExpLoads; u++) count_entry(bins[warp], lane, v[u], top);
                }
                for (; c < k; c += 32) count_entry(bins[warp], lane, p[c], top);
                SpreadScan scan;  // a level per lane
                for (int j = 0; j < kSpreadSteps / 2; j++) {
                    const unsigned w = bins[warp][j][lane];
                    scan.next(2 * j, __reduce_add_sync(0xffffffffu, (int)(w & 0xffffu)), k, lane);
                    scan.next(2 * j + 1, __reduce_add_sync(0xffffffffu, (int)(w >> 16)), k, lane);
                }
                const bool any = __any_sync(0xffffffffu, nonzero);
                if (lane >= 1 && lane <= kSpreadInts && any) atomicMax(&spread[lane - 1], scan.result(k, lane, top));
            }
        }
    } else {
        sum = sumsq_b;
        const int c = ((int)blockIdx.x - blocks_a) * 32 + lane;
        const bool col_ok = c < n;
        const bool sum_col = sum != nullptr && c < nv;
        int top = 0;
        double ss4[4] = {0.0, 0.0, 0.0, 0.0};  // a dependent FP64 FMA takes 64 cycles and more here
        if (col_ok) {
            int r = warp;
            for (; r + (kExpLoads - 1) * kExpWarps < k; r += kExpLoads * kExpWarps) {
                double v[kExpLoads];
#pragma unroll
                for (int u = 0; u < kExpLoads; u++) v[u] = load_now(B.row(z, r + u * kExpWarps) + c);
#pragma unroll
                for (int u = 0; u < kExpLoads; u++) {
                    top = max(top, exp_field(v[u]));
                    if (SUM && sum_col && r + u * kExpWarps < nv) ss4[u & 3] = fma(v[u], v[u], ss4[u & 3]);
                }
            }
            for (; r < k; r += kExpWarps) {
                const double v = B.row(z, r)[c];
                top = max(top, exp_field(v));
                if (SUM && sum_col && r < nv) ss4[0] = fma(v, v, ss4[0]);
            }
        }
        ss = (ss4[0] + ss4[1]) + (ss4[2] + ss4[3]);
        smax[warp][lane] = top;
        if constexpr (SPREAD) {
#pragma unroll
            for (int j = 0; j < kSpreadWords; j++) bins[warp][j][lane] = 0u;
            if (warp == 0) scount[lane][kSpreadSteps] = 0;
        }
        __syncthreads();
        top = 0;
#pragma unroll
        for (int w = 0; w < kExpWarps; w++) top = max(top, smax[w][lane]);
        if (warp == 0 && col_ok) eb[(int64_t)z * n + c] = top - 1022;
        if constexpr (SPREAD) {
            if (col_ok) {
                bool nonzero = top != 0;
                if (!nonzero)
                    for (int r = warp; r < k; r += kExpWarps) nonzero |= not_zero(B.row(z, r)[c]);
                int r = warp;
                for (; r + (kExpLoads - 1) * kExpWarps < k; r += kExpLoads * kExpWarps) {
                    double v[kExpLoads];
#pragma unroll
                    for (int u = 0; u < kExpLoads; u++) v[u] = load_now(B.row(z, r + u * kExpWarps) + c);
#pragma unroll
                    for (int u = 0; u < kExpLoads; u++) count_entry(bins[warp], lane, v[u], top);
                }
                for (; r < k; r += kExpWarps) count_entry(bins[warp], lane, B.row(z, r)[c], top);
                if (nonzero) scount[lane][kSpreadSteps] = 1;
            }
            __syncthreads();
            if (warp < kSpreadSteps / 2) {  // a word of bins per warp, a column per lane
                int lo = 0, hi = 0;
#pragma unroll
                for (int w = 0; w < kExpWarps; w++) {
                    const unsigned x = bins[w][warp][lane];
                    lo += (int)(x & 0xffffu);
                    hi += (int)(x >> 16);
                }
                scount[lane][2 * warp] = lo;
                scount[lane][2 * warp + 1] = hi;
            }
            __syncthreads();
            if (warp >= 1 && warp <= kSpreadInts) {  // a level per warp, a column per lane
                SpreadScan scan;
                for (int i = 0; i < kSpreadSteps; i++) scan.next(i, scount[lane][i], k, warp);
                const bool wanted = col_ok && scount[lane][kSpreadSteps];
                const int t = __reduce_max_sync(0xffffffffu, wanted ? scan.result(k, warp, top) : 0);
                if (lane == 0) atomicMax(&spread[kSpreadInts + warp - 1], t);
            }
        }
    }
    if (SUM && sum != nullptr) {  // the same for the whole block
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) ss += __shfl_down_sync(0xffffffffu, ss, off);
        if (lane == 0) ssum[warp] = ss;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < kExpWarps; w++) ss += ssum[w];
            if (ss != 0.0) atomicAdd(sum + (int64_t)z * sss, ss);
        }
    }
}

// --------------------------------------------------------- conversions --
// Each writes the planes' entries of 4 consecutive K positions.

__device__ __forceinline__ unsigned bf16_bits(float f) { return __bfloat16_as_ushort(__float2bfloat16_rn(f)); }

__device__ __forceinline__ void store4(uint16_t* dst, unsigned a, unsigned b, unsigned c, unsigned d) {
    *reinterpret_cast<uint2*>(dst) = make_uint2(a | (b << 16), c | (d << 16));
}

// hi = bf16(x), lo = bf16(x - hi) (three planes: hi, mid, lo), computed from
// xf = fp32(x), no FP64 operation (GB300's FP64 rate would bound this
// memory-bound pass); xf differs from x by 2^-24
// relative, far below what the three-product form keeps (~2^-16).
template <int PLANES>
struct ToBf16 {
    __device__ __forceinline__ void operator()(const double (&x)[4], int, uint16_t* dst, int64_t plane) const {
        float r[4];
#pragma unroll
        for (int u = 0; u < 4; u++) r[u] = f64_to_f32_rn(x[u]);
#pragma unroll
        for (int q = 0; q < PLANES; q++) {
            __nv_bfloat16 h[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                h[u] = __float2bfloat16_rn(r[u]);
                r[u] -= __bfloat162float(h[u]);  // exact in FP32
            }
            store4(dst + q * plane, __bfloat16_as_ushort(h[0]), __bfloat16_as_ushort(h[1]), __bfloat16_as_ushort(h[2]),
                   __bfloat16_as_ushort(h[3]));
        }
    }
};

// round(|x| 2^(b - e)), |x| < 2^e, ties away from zero: integer arithmetic on
// the IEEE fields.
__device__ __forceinline__ unsigned long long fixed_point(double x, int e, int b) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    int fe = (int)(u >> 52) & 0x7FF;
    unsigned long long m = u & ((1ull << 52) - 1);
    if (fe == 0)
        fe = 1;  // subnormal: no implicit bit
    else
        m |= 1ull << 52;
    const int sh = fe - 1075 + b - e;  // <= b - 53
    if (sh >= 0) return m << sh;
    return sh > -64 ? (m + (1ull << (-sh - 1))) >> (-sh) : 0ull;
}

// Fixed-point digits of x relative to 2^e (|x| < 2^e): N = round(|x| 2^(8s -
// 1 - e)) in balanced base 256 (low digits in [-128, 127], the top one in
// [-128, 128]), so x = 2^(e-7) sum_i d_i 2^(-8 i) to within half a unit of the
// last slice.
struct ToDigits {
    int planes;
    __device__ __forceinline__ void operator()(const double (&x)[4], int e, uint16_t* dst, int64_t plane) const {
        unsigned long long n[4];
        bool neg[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            n[u] = fixed_point(x[u], e, 8 * planes - 1);
            neg[u] = __double2hiint(x[u]) < 0;
        }
        for (int q = planes - 1; q >= 0; q--) {
            unsigned d[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                int v = q > 0 ? (int)(n[u] & 255u) : (int)n[u];
                if (q > 0) {
                    n[u] >>= 8;
                    if (v >= 128) {
                        v -= 256;
                        n[u] += 1;
                    }
                }
                d[u] = bf16_bits((float)(neg[u] ? -v : v));  // |d| <= 128: exact
            }
            store4(dst + q * plane, d[0], d[1], d[2], d[3]);
        }
    }
};

// Residues of the signed fixed-point integer: cut into PIECES balanced 14-bit
// pieces, each residue is one FP32 dot product of the pieces with the powers
// of 2^14 modulo p (every partial sum below 2^23, exact) minus p times the
// rounded quotient; |r| <= 128, exact in BF16.
constexpr int kPiece = 14;

__host__ __device__ constexpr int piece_weight(int l, int q) {  // 2^(14 q) modulo p, balanced
    const int p = crt_modulus(l);
    int v = 1;
    for (int i = 0; i < q; i++) v = v * (1 << kPiece) % p;
    return v > p / 2 ? v - p : v;
}

template <int PIECES>
struct ToResidues {
    int bits, moduli;
    __device__ __forceinline__ void operator()(const double (&x)[4], int e, uint16_t* dst, int64_t plane) const {
        float f[4][PIECES];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const unsigned long long n = fixed_point(x[u], e, bits);
            long long v = __double2hiint(x[u]) < 0 ? -(long long)n : (long long)n;
#pragma unroll
            for (int q = 0; q < PIECES; q++) {
                int d;
                if (q + 1 < PIECES) {
                    d = (int)((unsigned)v << (32 - kPiece)) >> (32 - kPiece);  // low 14 bits, signed
                    v = (v >> kPiece) + (d < 0 ? 1 : 0);  // (v - d) / 2^14; v - d may be 2^63 at 63 bits
                } else {
                    d = (int)v;
                }
                // d as FP32 without a conversion (16 per clock per SM): |d| < 2^22
                f[u][q] = __uint_as_float(0x4B400000u + (unsigned)d) - 12582912.0f;
            }
        }
#pragma unroll
        for (int l = 0; l < kCrtMaxModuli; l++) {
            if (l >= moduli) break;
            const float p = (float)crt_modulus(l), inv_p = 1.0f / (float)crt_modulus(l);
            unsigned r[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                float t = f[u][0];
#pragma unroll
                for (int q = 1; q < PIECES; q++) t = fmaf(f[u][q], (float)piece_weight(l, q), t);
                const float quot = fmaf(t, inv_p, 12582912.0f) - 12582912.0f;
                r[u] = __float_as_uint(fmaf(-quot, p, t));
            }
            // the high halves: the BF16 values (the rest of the words is zero)
            *reinterpret_cast<uint2*>(dst + l * plane) =
                make_uint2(__byte_perm(r[0], r[1], 0x7632), __byte_perm(r[2], r[3], 0x7632));
        }
    }
};

// --------------------------------------------------------------- kernel --

constexpr int kTileRows = 32, kTileK = 128;
constexpr int kTileLd = kTileK + 2;  // even: 16-byte reads

template <class Side, class Convert>
__global__ void __launch_bounds__(256)
split_kernel(Side A, Side B, const __grid_constant__ SplitTarget t, int64_t tiles_a, Convert convert,
             const int* active) {
    __shared__ __align__(16) double tile[kTileRows][kTileLd];
    const int z = blockIdx.y;
    if (!problem_on(active, z)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ktiles = (t.k + kTileK - 1) / kTileK;
    if ((int64_t)blockIdx.x < tiles_a) {
        const int64_t plane = (int64_t)t.rows * t.ld;
        uint16_t* dst = t.a + (int64_t)z * t.planes * plane;
        const int r0 = (int)(blockIdx.x / ktiles) * kTileRows, c = (int)(blockIdx.x % ktiles) * kTileK + 4 * lane;
        if (c >= t.k) return;
        auto load = [&](int r, double (&x)[4], int& e) {
            const double* p = A.row(z, t.row0 + r) + c;
            if (c + 3 < t.k && ((uintptr_t)p & 15u) == 0) {
                const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
                x[0] = a.x;
                x[1] = a.y;
                x[2] = b.x;
                x[3] = b.y;
            } else {
#pragma unroll
                for (int u = 0; u < 4; u++) x[u] = c + u < t.k ? p[u] : 0.0;
            }
            e = t.ea ? t.ea[(int64_t)z * t.m + t.row0 + r] : 0;
        };
        const int end = min(r0 + kTileRows, t.rows);
        double x[4], next[4];
        int e, next_e = 0;
        int r = r0 + warp;
        if (r < end) load(r, x, e);
#pragma unroll 1
        for (; r < end; r += 8) {
            if (r + 8 < end) load(r + 8, next, next_e);
            convert(x, e, dst + (int64_t)r * t.ld + c, plane);
#pragma unroll
            for (int u = 0; u < 4; u++) x[u] = next[u];
            e = next_e;
        }
        return;
    }
    const int64_t id = (int64_t)blockIdx.x - tiles_a;
    const int64_t plane = (int64_t)t.cols * t.ld;
    uint16_t* dst = t.b + (int64_t)z * t.planes * plane;
    // neighbouring blocks take neighbouring columns: whole lines of B
    const int ctiles = (t.cols + kTileRows - 1) / kTileRows;
    const int c0 = (int)(id % ctiles) * kTileRows, r0 = (int)(id / ctiles) * kTileK;
#pragma unroll 4
    for (int i = warp; i < kTileK; i += 8) {
        const int r = r0 + i, c = c0 + lane;
        tile[lane][i] = (r < t.k && c < t.cols) ? B.row(z, r)[t.col0 + c] : 0.0;
    }
    __syncthreads();
    const int r = r0 + 4 * lane;
    if (r >= t.k) return;
#pragma unroll 1
    for (int i = warp; i < kTileRows; i += 8) {
        const int c = c0 + i;
        if (c >= t.cols) break;
        const double2 a = *reinterpret_cast<const double2*>(&tile[i][4 * lane]);
        const double2 b = *reinterpret_cast<const double2*>(&tile[i][4 * lane + 2]);
        const double x[4] = {a.x, a.y, b.x, b.y};
        const int e = t.eb ? t.eb[(int64_t)z * t.n + t.col0 + c] : 0;
        convert(x, e, dst + (int64_t)c * t.ld + r, plane);
    }
}

template <class Side, class Convert>
int split_with(Side A, Side B, const SplitTarget& t, Convert c, int count, const int* active, cudaStream_t s) {
    const int64_t ktiles = (t.k + kTileK - 1) / kTileK;
    const int64_t ta = ktiles * ((t.rows + kTileRows - 1) / kTileRows), tb = ktiles * ((t.cols + kTileRows - 1) / kTileRows);
    if (ta + tb <= 0) return SPIN_OK;
    if (ta + tb > INT32_MAX) return SPIN_ERR_INVALID_ARG;
    split_kernel<Side, Convert><<<dim3((unsigned)(ta + tb), (unsigned)count), 256, 0, s>>>(A, B, t, ta, c, active);
    SPIN_CUDA_TRY(cudaGetLastError());
    return SPIN_OK;
}

template <class Side>
int split_sides(Side A, Side B, const SplitTarget& t, int count, const int* active, cudaStream_t s) {
    switch (t.kind) {
        case SPLIT_BF16:
            if (t.planes == 2) return split_with(A, B, t, ToBf16<2>(), count, active, s);
            if (t.planes == 3) return split_with(A, B, t, ToBf16<3>(), count, active, s);
            return SPIN_ERR_INVALID_ARG;
        case SPLIT_DIGITS:
            if (t.planes < 1 || t.planes > 7) return SPIN_ERR_INVALID_ARG;
            return split_with(A, B, t, ToDigits{t.planes}, count, active, s);
        default:
            if (t.planes < 1 || t.planes > kCrtMaxModuli || t.bits < 1 || t.bits > kCrtMaxBits)
                return SPIN_ERR_INVALID_ARG;
            static_assert(kCrtFewBits <= 4 * kPiece - 1, "pieces");
            if (t.bits <= kCrtFewBits)
                return split_with(A, B, t, ToResidues<4>{t.bits, t.planes}, count, active, s);
            return split_with(A, B, t, ToResidues<5>{t.bits, t.planes}, count, active, s);
    }
}

template <class Side>
int exponents_sides(Side A, Side B, const SplitSource& src, int m, int n, int k, int* ea, int* eb, double* sa,
                    double* sb, int* spread, int count, int64_t sss, cudaStream_t s) {
    const int ba = ea ? (m + kExpWarps - 1) / kExpWarps : 0, bb = eb ? (n + 31) / 32 : 0;
    if (ba + bb == 0) return SPIN_OK;
    const dim3 grid((unsigned)(ba + bb), (unsigned)count);
    auto kernel = sa != nullptr || sb != nullptr ? exponents_kernel<Side, false, true> : exponents_kernel<Side, false, false>;
    if constexpr (std::is_same<Side, SideOne>::value)
        if (spread != nullptr) kernel = exponents_kernel<Side, true, false>;
    kernel<<<grid, 32 * kExpWarps, 0, s>>>(A, B, m, n, k, ba, ea, eb, sa, sb, sss, spread, src.active, src.valid);
    SPIN_CUDA_TRY(cudaGetLastError());
    return SPIN_OK;
}

}  // namespace

int launch_exponents(const SplitSource& src, int m, int n, int k, int* ea, int* eb, double* sumsq_a, double* sumsq_b,
                     int* spread, cudaStream_t s) {
    if (src.count > 65535) return SPIN_ERR_INVALID_ARG;
    if (spread != nullptr && (src.count > 0 || sumsq_a != nullptr || sumsq_b != nullptr)) return SPIN_ERR_INVALID_ARG;
    if (src.count > 0)
        return exponents_sides(SideMany{src.Av}, SideMany{src.Bv}, src, m, n, k, ea, eb, sumsq_a, sumsq_b, spread,
                               src.count, 1, s);
    return exponents_sides(SideOne{src.A, src.lda}, SideOne{src.B, src.ldb}, src, m, n, k, ea, eb, sumsq_a, sumsq_b,
                           spread, 1, 0, s);
}

int launch_split(const SplitSource& src, const SplitTarget& t, cudaStream_t s) {
    if (src.count > 65535) return SPIN_ERR_INVALID_ARG;
    if (src.count > 0) return split_sides(SideMany{src.Av}, SideMany{src.Bv}, t, src.count, src.active, s);
    return split_sides(SideOne{src.A, src.lda}, SideOne{src.B, src.ldb}, t, 1, src.active, s);
}

}  // namespace spin
