// FP64-class products on the BF16 tensor cores by residues.
//
// The digit form (tc_gemm.cu, exact mode) cuts every operand into s digits
// and needs the s (s + 1) / 2 digit products of the leading weights.  Here
// the same fixed-point integers a' = round(a 2^(b - e)) (e the row's, for B
// the column's exponent) are taken modulo N pairwise coprime numbers p <=
// 256 instead, one product per modulus gives sum_k a'_ik b'_kj modulo p
// exactly, and the Chinese remainder theorem gives the whole sum, as long as
// the product of the moduli exceeds twice its largest magnitude (Ozaki,
// Uchino and Imamura, "Ozaki Scheme II", 2025, on INT8 units, whose rate on
// GB300 is far below BF16's).  Nothing is left out of the sum, and the number
// of tensor-core products falls from 21 to 13 or 14 for s = 6 (up to 15 above
// k = 32768), from 28 to 15 or 16 for s = 7 (17).
//
// Three kernels:
//   split    (split.cu) FP64 -> N BF16 planes of signed residues (|r| <= 128,
//            exact), six FP32 operations per residue, after a pass that takes
//            the exponents.
//   product  per modulus and 128 x 256 tile, exact FP32 runs of 1024 products
//            (|r r'| <= 2^14, sums <= 2^24) drained into int32, reduced
//            modulo p and written as one byte per output.  A tile of one
//            modulus is a work item of its own, so small products still fill
//            the SMs, and the drain is a conversion and an add per run.
//   combine  sum / P = frac(sum_l c_l u_l / p_l) with u_l the inverse of P /
//            p_l modulo p_l: one 96- or 128-bit fixed-point accumulation per
//            output with the constants u_l 2^128 / p_l (32-bit limbs, no
//            carries between moduli), then times P 2^(e + f - 2 b), rounded once to
//            FP64, and the product's epilogue (alpha, beta C, identity, sum of
//            squares).
// The integers are exact and every output depends on its row and column
// only, so the result does not depend on the panels the arena allows.
#include <math.h>
#include <string.h>

#include <utility>

#include <algorithm>

#include "crt.h"
#include "split.h"
#include "tc_pipe.cuh"

namespace spin {
namespace {

constexpr int kRunK = 1024;
constexpr int kMaxRuns = 96;  // 96 runs of 2^24 fit int32

// --------------------------------------------------------------- product --

struct CrtGemmParams {
    int M, N, K;        // of the panel pair
    int moduli, count;  // problems (>= 1)
    uint8_t* res;       // [z][modulus][M][ldr]
    int64_t ldr;        // a multiple of 16, >= N
    const int* active;
    int* err;
    unsigned p[kCrtMaxModuli], magic[kCrtMaxModuli], shift[kCrtMaxModuli];  // x + shift >= 0, a multiple of p
};

constexpr int kCrtBN = 256;
constexpr int kCrtEpiWarps = 16;
constexpr int kCrtHalf = kCrtBN / (kCrtEpiWarps / 4);  // columns per epilogue warp

// Persistent: one CTA per SM walks the items (problem, modulus, tile), the
// drain of one overlapping the next one's MMAs in the other TMEM accumulator.
// Warps as in tc_gemm_kernel: 0 TMA, 1 MMA, 2.. epilogue.
__global__ void __maxnreg__(Epi<kCrtEpiWarps>::MAXREG)
crt_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                const __grid_constant__ CrtGemmParams p) {
    // a problem switched off: nothing to set up (every thread reads the same flag)
    if (p.count == 1 && p.active != nullptr && p.active[0] == 0) return;
    constexpr int BN = kCrtBN, HALF = kCrtHalf;
    using C = Cfg<BN, 1>;
    constexpr int STAGES = C::STAGES;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* smA = base;
    unsigned char* smB = base + STAGES * A_TILE_BYTES;
    SmemCtl* ctl = reinterpret_cast<SmemCtl*>(base + STAGES * C::STAGE_BYTES);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int num_m = (p.M + BM - 1) / BM, num_n = (p.N + BN - 1) / BN;
    const int tiles = num_m * num_n;
    const int64_t items = (int64_t)p.count * p.moduli * tiles;
    // item t: plane (problem and modulus) zl and the tile's origin; tiles in
    // bands of GROUP_M row blocks, as in tc_gemm_kernel
    auto item_of = [&](int64_t t, int& zl, int& m0, int& n0) -> bool {
        zl = (int)(t / tiles);
        const int pid = (int)(t - (int64_t)zl * tiles);
        const int per_group = GROUP_M * num_n;
        const int first_m = (pid / per_group) * GROUP_M;
        const int gsize = min(num_m - first_m, GROUP_M);
        const int in_group = pid % per_group;
        m0 = (first_m + in_group % gsize) * BM;
        n0 = (in_group / gsize) * BN;
        return p.active == nullptr || p.active[zl / p.moduli] != 0;
    };
    const int KB = (p.K + BK - 1) / BK;
    constexpr int run_kb = kRunK / BK;
    const int runs = (KB + run_kb - 1) / run_kb;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; s++) {
            mbar_init(&ctl->full[s], 1);
            mbar_init(&ctl->empty[s], 1);
        }
        for (int b = 0; b < 2; b++) {
            mbar_init(&ctl->tfull[b], 1);
            mbar_init(&ctl->tempty[b], kCrtEpiWarps);
        }
        mbar_init(&ctl->final_bar, 1);
        ctl->abort = 0;
        fence_mbar_init();
        prefetch_tensormap(&tmA);
        prefetch_tensormap(&tmB);
    }
    if (warp == 1) {
        tmem_alloc(&ctl->tmem_base, 2 * BN);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    volatile int* abort = &ctl->abort;

    if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            int zl, m0, n0;
            for (int64_t t = blockIdx.x; t < items && ok; t += gridDim.x) {
                if (!item_of(t, zl, m0, n0)) continue;
                const int ya = zl * p.M + m0, yb = zl * p.N + n0;
                for (int kb = 0; kb < KB; kb++) {
                    const int s = it % STAGES;
                    ok = mbar_wait(&ctl->empty[s], (uint32_t)((it / STAGES) & 1) ^ 1u, abort, WAIT_LIMIT_NS);
                    if (!ok) break;
                    mbar_arrive_expect_tx(&ctl->full[s], C::STAGE_BYTES);
                    tma_load_2d(smA + s * A_TILE_BYTES, &tmA, kb * BK, ya, &ctl->full[s]);
                    tma_load_2d(smB + s * C::B_TILE_BYTES, &tmB, kb * BK, yb, &ctl->full[s]);
                    it++;
                }
            }
            if (!ok) raise_timeout(ctl, p.err);
            // own copies still in flight: the last min(STAGES, it) loads
            for (int j = max(0, it - STAGES); j < it; j++) {
                volatile int never = 0;
                mbar_wait(&ctl->full[j % STAGES], (uint32_t)((j / STAGES) & 1), &never, WAIT_LIMIT_NS);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16_f32(BM, BN);
            int it = 0, run = 0;
            bool ok = true;
            int zl, m0, n0;
            for (int64_t t = blockIdx.x; t < items && ok; t += gridDim.x) {
                if (!item_of(t, zl, m0, n0)) continue;
                for (int kb = 0; kb < KB && ok;) {
                    const int buf = run & 1;
                    ok = mbar_wait(&ctl->tempty[buf], (uint32_t)((run >> 1) & 1) ^ 1u, abort, WAIT_LIMIT_NS);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d = tmem_base + (uint32_t)(buf * BN);
                    const int kb0 = kb, kb1 = min(KB, kb + run_kb);
                    for (; kb < kb1; kb++) {
                        const int s = it % STAGES;
                        ok = mbar_wait(&ctl->full[s], (uint32_t)((it / STAGES) & 1), abort, WAIT_LIMIT_NS);
                        if (!ok) break;
                        tc_fence_after();
                        const uint64_t ad = sdesc_kmajor_sw128(smem_u32(smA + s * A_TILE_BYTES));
                        const uint64_t bd = sdesc_kmajor_sw128(smem_u32(smB + s * C::B_TILE_BYTES));
#pragma unroll
                        for (int k = 0; k < BK / 16; k++)
                            mma_bf16(d, ad + ((k * 32) >> 4), bd + ((k * 32) >> 4), idesc, (kb == kb0 && k == 0) ? 0u : 1u);
                        mma_commit(&ctl->empty[s]);
                        it++;
                    }
                    if (ok) mma_commit(&ctl->tfull[buf]);
                    run++;
                }
            }
            if (!ok) raise_timeout(ctl, p.err);
            // every MMA issued so far has completed once final_bar flips
            mma_commit(&ctl->final_bar);
            volatile int never = 0;
            mbar_wait(&ctl->final_bar, 0u, &never, WAIT_LIMIT_NS);
        }
        __syncwarp();
    } else {
        const int quarter = warp & 3;       // TMEM lane quarter this warp may access
        const int half = (warp - 2) >> 2;   // column group of the tile
        const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * HALF);
        int run = 0;
        int zl, m0, n0;
        bool ok = true;
        for (int64_t t = blockIdx.x; t < items && ok; t += gridDim.x) {
            if (*abort) break;
            if (!item_of(t, zl, m0, n0)) continue;
            // columns (of this warp's HALF) and rows that exist
            const int row = m0 + quarter * 32 + lane, col0 = n0 + half * HALF;
            const int ncol = m0 + quarter * 32 < p.M ? min(HALF, p.N - col0) : 0;
            int acc[HALF];
            for (int c = 0; c < runs && ok; c++) {
                const int buf = run & 1;
                ok = mbar_wait(&ctl->tfull[buf], (uint32_t)((run >> 1) & 1), abort, WAIT_LIMIT_NS);
                if (!ok) {
                    raise_timeout(ctl, p.err);
                    break;
                }
                tc_fence_after();
#pragma unroll
                for (int c0 = 0; c0 < HALF; c0 += 16) {
                    if (c0 >= ncol) break;
                    uint32_t v[16];
                    tmem_ld_32x32b_x16(lane_addr + (uint32_t)(buf * BN + c0), v);
                    tmem_ld_wait();
                    if (c == 0) {
#pragma unroll
                        for (int j = 0; j < 16; j++) acc[c0 + j] = __float2int_rn(__uint_as_float(v[j]));
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; j++) acc[c0 + j] += __float2int_rn(__uint_as_float(v[j]));
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&ctl->tempty[buf]);
                run++;
            }
            if (!ok) break;
            if (row < p.M) {
                const int l = zl % p.moduli;
                const unsigned mod = p.p[l], magic = p.magic[l], shift = p.shift[l];
                uint8_t* out = p.res + ((int64_t)zl * p.M + row) * p.ldr + col0;
#pragma unroll
                for (int c0 = 0; c0 < HALF; c0 += 16) {
                    if (c0 >= ncol) break;
                    uint32_t w[4];
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        uint32_t b[4];
#pragma unroll
                        for (int j = 0; j < 4; j++) {
                            const unsigned u = (unsigned)acc[c0 + 4 * q + j] + shift;
                            const unsigned r = u - __umulhi(u, magic) * mod;  // in [0, 2 mod)
                            b[j] = min(r, r - mod);
                        }
                        w[q] = __byte_perm(__byte_perm(b[0], b[1], 0x0040), __byte_perm(b[2], b[3], 0x0040), 0x5410);
                    }
                    *reinterpret_cast<uint4*>(out + c0) = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 2 * BN);
    }
}

// --------------------------------------------------------------- combine --

struct CrtTable {
    unsigned v[kCrtMaxModuli][4];  // u_l 2^128 / p_l modulo 2^128, low limb first
    unsigned long long pm;         // the product of the moduli = pm 2^pe, 2^63 <= pm < 2^64
    int pe;
    int moduli, bits;
};

// The sum whose residue fraction (sum / P modulo 1) has the limbs w, lowest
// first, times 2^scale, rounded to FP64 (neg: times -1).
template <int LIMBS>
__device__ __forceinline__ double crt_value(unsigned (&w)[LIMBS], const CrtTable& t, int scale, bool neg) {
    const unsigned flip = (unsigned)((int)w[LIMBS - 1] >> 31);  // the symmetric range: fractions of
    unsigned carry = flip & 1u;                                 // one half and more are negative
    unsigned any = 0u;
#pragma unroll
    for (int i = 0; i < LIMBS; i++) {
        const unsigned x = (w[i] ^ flip) + carry;
        carry = x < carry ? 1u : 0u;
        w[i] = x;
        any |= x;
    }
    if (any == 0u) return 0.0;
    int lz = 0;  // bits before the first set one, below 32 but for sums of under 2^-32 P
    while (w[LIMBS - 1] == 0u) {
#pragma unroll
        for (int i = LIMBS - 1; i > 0; i--) w[i] = w[i - 1];
        w[0] = 0u;
        lz += 32;
    }
    const int s = __clz((int)w[LIMBS - 1]);
    lz += s;
    const unsigned h1 = __funnelshift_l(w[LIMBS - 2], w[LIMBS - 1], s), h0 = __funnelshift_l(w[LIMBS - 3], w[LIMBS - 2], s);
    unsigned long long prod = __umul64hi((unsigned long long)h1 << 32 | h0, t.pm);  // the sum = prod 2^(pe - lz)
    const int one = (int)(~prod >> 63);                                             // prod >= 2^62
    if (one) prod += prod;
    const unsigned long long m = (prod >> 11) + ((prod >> 10) & 1ull);  // 53 bits, or 2^53
    const int e = 11 + t.pe - lz - one + scale;                         // value = m 2^e
    const int be = e + 52 + 1023;
    const unsigned long long sign = (unsigned long long)(neg != (flip != 0u)) << 63;
    if (be >= 1 && be <= 2045)
        return __longlong_as_double((long long)((((unsigned long long)(be - 1) << 52) + m) | sign));
    double v;  // where it stands: not computed for everyone and selected afterwards
    asm volatile("cvt.rn.f64.u64 %0, %1;" : "=d"(v) : "l"(m));
    return __longlong_as_double(__double_as_longlong(ldexp(v, e)) | (long long)sign);
}

// 4 columns of a row per thread.  p: the whole product (views, epilogue);
// (row0, col0): the panel pair's origin; rows x cols its size.  LIMBS 32-bit
// limbs of the fraction: 3 leave an error of 2^-84 P, i.e. below 2^-75 k of the
// largest entries' product for the formats that use it (bits <= 55, P at most
// 2^9 times the least for them).
// Bound by instructions (about 200 per output, 39 to 80 of them 32 x 32 + 64
// bit multiply-adds): the number of moduli is a template argument, so the words
// of a thread's four outputs (and of C) are all requested before the first is
// used and the constants are immediate; SUM (the sum of squares) is one as well,
// as the compiler computes squares nobody asked for on the FP64 pipe.  4096^2
// outputs of 15 moduli with C: 169 us (16: 173), 187 without SUM apart, 344 with four words
// in flight in a run-time loop and the indices by a division each (540 MB: 80
// us).  Four blocks an SM spill: 64 registers.
template <int LIMBS, int MODULI, bool SUM>
__global__ void __launch_bounds__(256, 2)
crt_combine_kernel(const uint8_t* __restrict__ res, int64_t ldr, int rows, int cols, int row0, int col0,
                   const __grid_constant__ CrtTable t, const __grid_constant__ TcGemmParams p) {
    const int z = blockIdx.z;
    if (p.active != nullptr && p.active[p.batch ? z : 0] == 0) return;
    const int64_t plane = (int64_t)rows * ldr;
    res += (int64_t)z * MODULI * plane;
    const int* row_exp = p.row_exp + (int64_t)z * p.M + row0;
    const int* col_exp = p.col_exp + (int64_t)z * p.N + col0;
    const int groups = (cols + 3) / 4;
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    const int dr = (int)(stride / groups), dc = (int)(stride % groups);
    const int so = p.sum_order ? p.sum_order[z] : 0x7fffffff;
    // alpha = +-1, beta = 0 or 1, told apart by their bits: an FP64 compare is
    // made again for every output
    const bool add = (unsigned)__double2hiint(p.beta) << 1 != 0u, minus = __double2hiint(p.alpha) < 0;
    double ss = 0.0, ss2 = 0.0;
    int cg = (int)(first % groups);
    for (int64_t rr = first / groups; rr < rows; rr += dr) {
        const int r = (int)rr, c = cg * 4;
        cg += dc;
        if (cg >= groups) {
            cg -= groups;
            rr++;
        }
        const uint8_t* src = res + (int64_t)r * ldr + c;
        unsigned word[MODULI];
#pragma unroll
        for (int l = 0; l < MODULI; l++) word[l] = *reinterpret_cast<const unsigned*>(src + l * plane);
        const int er = row_exp[r], grow = row0 + r;
        const double* crow = add ? in_row(p, z, grow) + col0 + c : nullptr;
        double* drow = out_row(p, z, grow) + col0 + c;
        // whole 32-byte sectors where the views allow it
        const bool quad = c + 3 < cols && aligned32(drow) && (!add || aligned32(crow));
        double old[4];
        if (add) {
            if (quad) {
                ld_global_v4(crow, old);
            } else {
#pragma unroll
                for (int u = 0; u < 4; u++) old[u] = c + u < cols ? crow[u] : 0.0;
            }
        }
        double val[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            unsigned long long acc[LIMBS] = {};
#pragma unroll
            for (int l = 0; l < MODULI; l++) {
                const unsigned b = (word[l] >> (8 * u)) & 255u;
#pragma unroll
                for (int i = 0; i < LIMBS; i++) acc[i] += (unsigned long long)b * t.v[l][4 - LIMBS + i];
            }
            const int ec = c + u < cols ? col_exp[c + u] : 0;
            unsigned w[LIMBS];  // the limbs, carried
            unsigned long long carry = 0ull;
#pragma unroll
            for (int i = 0; i < LIMBS; i++) {
                carry += acc[i];
                w[i] = (unsigned)carry;
                carry >>= 32;
            }
            val[u] = crt_value<LIMBS>(w, t, er + ec - 2 * t.bits, minus);
            // an infinity or NaN in the row or column (no fixed point has it)
            if (er > 1024 || ec > 1024) val[u] = __longlong_as_double(0x7ff8000000000000ll);
        }
        const int gcol = col0 + c;
        if (add) {  // beta = 1
#pragma unroll
            for (int u = 0; u < 4; u++) val[u] = add_now(old[u], val[u]);
        }
        if (p.add_identity && (unsigned)(grow - gcol) < 4u) {
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (gcol + u == grow) val[u] = add_now(val[u], 1.0);
        }
        if (SUM && grow < so) {
            if (c + 3 < cols && gcol + 3 < so) {
                ss = fma(val[0], val[0], ss);
                ss2 = fma(val[1], val[1], ss2);
                ss = fma(val[2], val[2], ss);
                ss2 = fma(val[3], val[3], ss2);
            } else {
#pragma unroll
                for (int u = 0; u < 4; u++)
                    if (gcol + u < so && c + u < cols) ss = fma(val[u], val[u], ss);
            }
        }
        if (quad) {
            st_global_v4(drow, val);
        } else {
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (c + u < cols) drow[u] = val[u];
        }
    }
    if (SUM) {
        __shared__ double part[8];
        ss += ss2;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) ss += __shfl_down_sync(0xffffffffu, ss, off);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = ss;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int i = 1; i < 8; i++) ss += part[i];
            if (ss != 0.0) atomicAdd(p.sumsq + (p.batch ? z : 0), ss);
        }
    }
}

// ------------------------------------------------------------------ host --

using CombineKernel = void (*)(const uint8_t*, int64_t, int, int, int, int, CrtTable, TcGemmParams);
template <int LIMBS, bool SUM, int FIRST, int... M>
CombineKernel combine_of(int moduli, std::integer_sequence<int, M...>) {
    static constexpr CombineKernel kernels[] = {crt_combine_kernel<LIMBS, FIRST + M, SUM>...};
    return moduli >= FIRST && moduli < FIRST + (int)sizeof...(M) ? kernels[moduli - FIRST] : nullptr;
}
// For k <= 98304: 31 to 55 bits take 8 to 17 moduli, 63 bits 17 to 19 (large
// FP64 products, which have no sum of squares).
CombineKernel combine_kernel(const CrtFormat& f, bool sum) {
    const auto few = std::make_integer_sequence<int, 18 - kCrtMinModuli>();
    const auto many = std::make_integer_sequence<int, kCrtMaxModuli - 16>();
    if (f.bits <= kCrtFewBits)
        return sum ? combine_of<3, true, kCrtMinModuli>(f.moduli, few) : combine_of<3, false, kCrtMinModuli>(f.moduli, few);
    return sum ? nullptr : combine_of<4, false, 17>(f.moduli, many);
}

// floor(2^128 u / p) with p, u < 2^9, rounded, as four limbs.
void fraction_limbs(unsigned u, unsigned p, unsigned (&v)[4]) {
    unsigned rem = u % p;
    unsigned q[5];  // 32-bit digits of u / p behind the point, one more for the rounding
    for (int i = 0; i < 5; i++) {
        const unsigned long long t = (unsigned long long)rem << 32;
        q[i] = (unsigned)(t / p);
        rem = (unsigned)(t % p);
    }
    unsigned carry = q[4] >> 31;
    for (int i = 3; i >= 0; i--) {
        const unsigned long long t = (unsigned long long)q[i] + carry;
        v[3 - i] = (unsigned)t;
        carry = (unsigned)(t >> 32);
    }
}

void crt_table(const CrtFormat& f, CrtTable* t) {
    // P as a little-endian multi-limb integer (at most 160 bits)
    unsigned limb[6] = {1, 0, 0, 0, 0, 0};
    for (int l = 0; l < f.moduli; l++) {
        unsigned long long carry = 0;
        for (unsigned& x : limb) {
            const unsigned long long s = (unsigned long long)x * (unsigned)crt_modulus(l) + carry;
            x = (unsigned)s;
            carry = s >> 32;
        }
    }
    int top = 191;
    while (top > 0 && !((limb[top / 32] >> (top % 32)) & 1u)) top--;
    t->pm = 0;
    for (int i = 0; i < 64; i++) {
        const int bit = top - i;
        t->pm = (t->pm << 1) | (bit >= 0 ? (limb[bit / 32] >> (bit % 32)) & 1u : 0u);
    }
    if (top >= 64 && ((limb[(top - 64) / 32] >> ((top - 64) % 32)) & 1u) && t->pm != ~0ull) t->pm++;
    t->pe = top - 63;
    for (int l = 0; l < f.moduli; l++) {
        const unsigned p = (unsigned)crt_modulus(l);
        unsigned rest = 1 % p;
        for (int k = 0; k < f.moduli; k++)
            if (k != l) rest = rest * (unsigned)crt_modulus(k) % p;
        unsigned u = 1;
        while (rest * u % p != 1 % p) u++;
        fraction_limbs(u, p, t->v[l]);
    }
    t->moduli = f.moduli;
    t->bits = f.bits;
}

constexpr int kMaxPanels = 64;
size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

struct CrtPanels {
    int64_t rows, cols;  // of a panel pair
    int64_t ld, ldr;
    size_t off_a, off_b, off_res, total;
};

CrtPanels panel_layout(int64_t m, int64_t n, int64_t k, int moduli, int64_t count, int64_t rows, int64_t cols) {
    CrtPanels c;
    c.rows = std::min(rows, m);
    c.cols = std::min(cols, n);
    c.ld = tc_ld(k);
    c.ldr = (int64_t)round_up((size_t)c.cols, 16);
    c.off_a = 256 + round_up((size_t)(count * (m + n)) * sizeof(int), 256);  // 256: alignment of the arena
    c.off_b = c.off_a + round_up((size_t)(count * moduli * c.rows * c.ld) * 2, 256);
    c.off_res = c.off_b + round_up((size_t)(count * moduli * c.cols * c.ld) * 2, 256);
    c.total = c.off_res + round_up((size_t)(count * moduli * c.rows * c.ldr), 256);
    return c;
}

// A p-th of x, in whole tiles unless a panel is smaller than one.
int64_t panel_size(int64_t x, int64_t p, int64_t tile) {
    const size_t part = (size_t)((x + p - 1) / p);
    return (int64_t)round_up(part, part > (size_t)tile ? (size_t)tile : 16);
}

// Panels that fit: A's rows once per row panel, B's columns once per row
// panel and column panel.  The cheapest by the elements split (about 6 ps
// each and modulus-proportional) and launches.
bool choose_panels(int64_t m, int64_t n, int64_t k, int moduli, int64_t count, size_t bytes, CrtPanels* best) {
    double least = 1e300;
    for (int pa = 1; pa <= kMaxPanels; pa++) {
        const int64_t rows = panel_size(m, pa, BM);
        if (pa > 1 && rows >= panel_size(m, pa - 1, BM)) continue;
        for (int pb = 1; pb <= kMaxPanels; pb++) {
            const int64_t cols = panel_size(n, pb, kCrtBN);
            const CrtPanels c = panel_layout(m, n, k, moduli, count, rows, cols);
            if (c.total > bytes) continue;
            const double na = (double)((m + rows - 1) / rows), nb = (double)((n + cols - 1) / cols);
            const double cost = na * (double)n * (double)k * (double)count * 6e-12 + na * nb * 15e-6;
            if (cost < least) {
                least = cost;
                *best = c;
            }
            break;  // fewer columns only cost more
        }
    }
    return least < 1e300;
}

int crt_run(const CrtProduct& p, const CrtFormat& f, const CrtPanels& c, unsigned char* arena, cudaStream_t s,
            int* launches) {
    const int count = p.count > 0 ? p.count : 1;
    const int m = (int)p.m, n = (int)p.n, k = (int)p.k;
    int* ea = p.a_exps_out != nullptr ? p.a_exps_out : (int*)arena;
    int* eb = (int*)arena + (size_t)count * (size_t)m;
    uint16_t* pa = (uint16_t*)(arena + c.off_a - 256);
    uint16_t* pb = (uint16_t*)(arena + c.off_b - 256);
    uint8_t* res = arena + c.off_res - 256;
    int nl = 0;
    SplitSource src;
    src.count = p.count;
    src.A = p.A;
    src.lda = p.lda;
    src.B = p.B;
    src.ldb = p.ldb;
    src.Av = p.Av;
    src.Bv = p.Bv;
    src.active = p.active;
    src.valid = p.valid;
    const bool known = p.a_exps != nullptr;
    if (known) ea = const_cast<int*>(p.a_exps);
    if (p.b_exps != nullptr) eb = const_cast<int*>(p.b_exps);
    int rc = SPIN_OK;
    if (!known || p.b_exps == nullptr) {
        rc = launch_exponents(src, m, n, k, known ? nullptr : ea, eb, p.sumsq_a, p.sumsq_b, nullptr, s);
        if (rc) return rc;
        nl++;
    }

    CrtTable table;
    crt_table(f, &table);
    TcGemmParams q = {};
    q.M = m;
    q.N = n;
    q.K = k;
    q.alpha = p.alpha;
    q.beta = p.beta;
    q.C = p.C;
    q.ldc = p.ldc;
    q.D = p.D;
    q.ldd = p.ldd;
    q.row_exp = ea;
    q.col_exp = eb;
    q.add_identity = p.add_identity;
    q.sumsq = p.sumsq_d;
    q.active = p.active;
    q.sum_order = p.valid;
    if (p.count > 0) {
        q.batch = p.count;
        q.c_base = p.beta != 0.0 ? p.Cv.base : nullptr;
        q.c_lds = p.Cv.lds;
        q.c_ld = p.Cv.ld;
        q.c_r0 = p.Cv.r0;
        q.c_c0 = p.Cv.c0;
        q.d_base = const_cast<double* const*>(p.Dv.base);
        q.d_lds = p.Dv.lds;
        q.d_ld = p.Dv.ld;
        q.d_r0 = p.Dv.r0;
        q.d_c0 = p.Dv.c0;
    }
    CrtGemmParams g = {};
    g.K = k;
    g.moduli = f.moduli;
    g.count = count;
    g.res = res;
    g.active = p.active;
    g.err = p.err;
    for (int l = 0; l < f.moduli; l++) {
        g.p[l] = (unsigned)crt_modulus(l);
        g.magic[l] = (unsigned)((1ull << 32) / g.p[l]);
        g.shift[l] = 0x80000000u / g.p[l] * g.p[l];
    }
    constexpr size_t smem = Cfg<kCrtBN, 1>::SMEM_BYTES;
    static PerDeviceOnce attrs;
    rc = attrs.run([&]() -> int {
        SPIN_CUDA_TRY(cudaFuncSetAttribute(crt_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        return SPIN_OK;
    });
    if (rc) return rc;
    const int sms = sm_count();
    const CombineKernel combine = combine_kernel(f, q.sumsq != nullptr);
    if (combine == nullptr) return SPIN_ERR_INVALID_ARG;
    for (int row0 = 0; row0 < m; row0 += (int)c.rows) {
        const int rows = std::min((int)c.rows, m - row0);
        CUtensorMap ta;
        if ((rc = make_map(&ta, pa, k, (int64_t)count * f.moduli * rows, c.ld, BM))) return rc;
        for (int col0 = 0; col0 < n; col0 += (int)c.cols) {
            const int cols = std::min((int)c.cols, n - col0);
            // the row panel's planes with its first column panel; a lone
            // column panel's planes are still there from the first row panel
            SplitTarget t{SPLIT_RESIDUES, f.moduli, f.bits, m, n, k, row0, col0 == 0 ? rows : 0, col0, cols, ea, eb, pa,
                          pb, c.ld};
            if (row0 > 0 && c.cols >= n) t.cols = 0;
            if ((rc = launch_split(src, t, s))) return rc;
            nl++;
            CUtensorMap tb;
            if ((rc = make_map(&tb, pb, k, (int64_t)count * f.moduli * cols, c.ld, kCrtBN))) return rc;
            g.M = rows;
            g.N = cols;
            g.ldr = (int64_t)round_up((size_t)cols, 16);
            const int64_t items =
                (int64_t)((rows + BM - 1) / BM) * ((cols + kCrtBN - 1) / kCrtBN) * f.moduli * count;
            crt_gemm_kernel<<<(unsigned)std::min<int64_t>(items, sms), Epi<kCrtEpiWarps>::THREADS, smem, s>>>(ta, tb, g);
            SPIN_CUDA_TRY(cudaGetLastError());
            const int64_t total = (int64_t)rows * ((cols + 3) / 4);
            const int64_t per = std::max<int64_t>(1, (int64_t)sms * 8 / count);
            const dim3 cg((unsigned)std::min<int64_t>((total + 255) / 256, per), 1, (unsigned)count);
            combine<<<cg, 256, 0, s>>>(res, g.ldr, rows, cols, row0, col0, table, q);
            SPIN_CUDA_TRY(cudaGetLastError());
            nl += 2;
        }
    }
    if (launches) *launches += nl;
    return SPIN_OK;
}

}  // namespace

CrtFormat crt_format(int64_t k, int min_bits) {
    CrtFormat f{0, 0};
    if (k < 1 || k > (int64_t)kMaxRuns * kRunK) return f;
    double log2p = 0.0;
    for (int l = 0; l < kCrtMaxModuli; l++) {
        log2p += std::log2((double)crt_modulus(l));
        // P > 2 k 2^(2 bits); the margin covers the logarithms' rounding
        const int bits = (int)std::floor((log2p - 1.0 - std::log2((double)k) - 1e-9) / 2.0);
        if (bits >= min_bits) {
            f.moduli = l + 1;
            f.bits = std::min(bits, min_bits <= kCrtFewBits ? kCrtFewBits : kCrtMaxBits);
            return f;
        }
    }
    return f;
}

size_t crt_full_bytes(int64_t m, int64_t n, int64_t k, int moduli, int count) {
    return panel_layout(m, n, k, moduli, std::max(count, 1), m, n).total;
}

size_t crt_min_bytes(int64_t m, int64_t n, int64_t k, int moduli, int count) {
    return panel_layout(m, n, k, moduli, std::max(count, 1), panel_size(m, kMaxPanels, BM),
                        panel_size(n, kMaxPanels, kCrtBN))
        .total;
}

namespace {

BatchView skip(BatchView v, int z) {
    v.base += z;
    if (v.lds) v.lds += z;
    return v;
}

}  // namespace

int crt_product(const CrtProduct& p, void* arena, size_t bytes, cudaStream_t s, int* launches) {
    if (p.m <= 0 || p.n <= 0) return SPIN_OK;
    if (p.count < 0 || p.count > 65535) return SPIN_ERR_INVALID_ARG;
    if (!(p.alpha == 1.0 || p.alpha == -1.0) || !(p.beta == 0.0 || p.beta == 1.0)) return SPIN_ERR_INVALID_ARG;
    const CrtFormat f = crt_format(p.k, p.min_bits);
    if (f.moduli == 0) return SPIN_ERR_INVALID_ARG;
    unsigned char* base = (unsigned char*)round_up((size_t)(uintptr_t)arena, 256);
    CrtPanels c;
    if (p.count == 0) {
        if (!choose_panels(p.m, p.n, p.k, f.moduli, 1, bytes, &c)) return SPIN_ERR_INVALID_ARG;
        if (f.moduli * std::max(c.rows, c.cols) > INT32_MAX) return SPIN_ERR_INVALID_ARG;  // TMA row coordinate
        return crt_run(p, f, c, base, s, launches);
    }
    // as many problems at a time as the arena (and the TMA row coordinate)
    // holds whole, the same number each time; in panels, one at a time, if none
    const auto fits = [&](int64_t z) {
        return crt_full_bytes(p.m, p.n, p.k, f.moduli, (int)z) <= bytes &&
               z * f.moduli * std::max(p.m, p.n) <= INT32_MAX;
    };
    int most = p.count;
    if (!fits(most)) {
        int lo = 0;  // fits, or none
        while (most - lo > 1) {
            const int mid = lo + (most - lo) / 2;
            if (fits(mid))
                lo = mid;
            else
                most = mid;
        }
        most = std::max(lo, 1);
    }
    const int chunks = (p.count + most - 1) / most, step = (p.count + chunks - 1) / chunks;
    for (int z = 0; z < p.count; z += step) {
        CrtProduct q = p;
        q.count = std::min(step, p.count - z);
        q.Av = skip(p.Av, z);
        q.Bv = skip(p.Bv, z);
        if (p.beta != 0.0) q.Cv = skip(p.Cv, z);
        q.Dv = skip(p.Dv, z);
        if (p.active) q.active = p.active + z;
        if (p.valid) q.valid = p.valid + z;
        if (p.sumsq_a) q.sumsq_a = p.sumsq_a + z;
        if (p.sumsq_b) q.sumsq_b = p.sumsq_b + z;
        if (p.sumsq_d) q.sumsq_d = p.sumsq_d + z;
        if (p.a_exps) q.a_exps = p.a_exps + (int64_t)z * p.m;
        if (p.b_exps) q.b_exps = p.b_exps + (int64_t)z * p.n;
        if (p.a_exps_out) q.a_exps_out = p.a_exps_out + (int64_t)z * p.m;
        if (!choose_panels(q.m, q.n, q.k, f.moduli, q.count, bytes, &c)) return SPIN_ERR_INVALID_ARG;
        const int rc = crt_run(q, f, c, base, s, launches);
        if (rc) return rc;
    }
    return SPIN_OK;
}

}  // namespace spin
