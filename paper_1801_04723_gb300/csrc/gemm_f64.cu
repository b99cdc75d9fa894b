// FP64 level products of the plain method: D = beta*C + alpha*(A B).
//
// Algorithm 1's six products per recursion level (II, III, IV, C12, C21,
// VII; Sec. 3.1) and its two subtractions (V = IV - A22, C11 = I - VII) are
// one kernel here: the subtraction and the sign are the epilogue.
//
// On GB300 the FP64 pipe retires about 2 FMA per clock per SM (DFMA measured
// at ~1.2 TFLOP/s over 152 SMs; DMMA at ~1.05-1.10), so the kernel is
// bounded by the FP64 pipe at any reasonable tiling, and a product runs at
// the rate of the SMs it occupies.  A 64x64 output tile per 256-thread CTA,
// 4x4 register tile per thread, k-step 16 staged through double-buffered
// shared memory, gives 16 independent FMAs per thread per k-slice and needs
// ~0.25 B of L2 traffic per FMA -- far under any memory roof.  Where the last
// wave of 64x64 tiles would leave SMs idle (most products of a few hundred to
// a few thousand rows) a product takes 32x32, 16x16, 8x16 or 8x8 tiles
// instead.  Every output is one FMA chain over k in order, whatever
// the tile, so the tile size never changes a result bit.  Operands are
// arbitrary strided views (no alignment beyond 8 B).
#include <math.h>
#include <stdlib.h>

#include <cmath>

#include "common.cuh"

namespace spin {
namespace {

constexpr int BK = 16, NT = 256;
// Tile rows per group of the single-product tile order.  Measured on a
// 4096^3 product (ncu dram__bytes_read.sum + dram__bytes_write.sum, same
// duration every time): 3.87 GB in row-major order, 1.49 GB with groups of
// 8 tile rows, 1.03 GB with 16, against 0.40 GB of operands and result.
constexpr int kTileGroup = 16;

// One TM x TM output tile per 256-thread CTA: thread (tx, ty) of a 16 x 16
// grid owns a (TM/16) x (TM/16) register tile.
template <int TM>
__device__ __forceinline__ void gemm_f64_tile(int64_t m, int64_t n, int64_t k, double alpha,
                                              const double* __restrict__ A, int64_t lda,
                                              const double* __restrict__ B, int64_t ldb, double beta,
                                              const double* C, int64_t ldc, double* D, int64_t ldd,
                                              int64_t tile_m, int64_t tile_n) {
    constexpr int T = TM / 16;        // outputs per thread along each side
    constexpr int BR = NT / TM;       // B tile rows loaded per pass
    __shared__ double As[2][BK][TM + 1];
    __shared__ double Bs[2][BK][TM];
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int64_t m0 = tile_m * TM, n0 = tile_n * TM;

    // load mapping: A tile (TM x BK): row = ty + 16*i, kk = tx; B tile (BK x TM): kr = tid/TM + BR*i, col = tid%TM
    const int a_kk = tx;
    const int b_col = tid % TM, b_kr = tid / TM;
    double ra[T], rb[T];

    auto load_regs = [&](int64_t k0) {
#pragma unroll
        for (int i = 0; i < T; i++) {
            const int64_t r = m0 + ty + 16 * i, c = k0 + a_kk;
            ra[i] = (r < m && c < k) ? A[r * lda + c] : 0.0;
            const int64_t kr = k0 + b_kr + BR * i, cc = n0 + b_col;
            rb[i] = (kr < k && cc < n) ? B[kr * ldb + cc] : 0.0;
        }
    };
    auto store_smem = [&](int buf) {
#pragma unroll
        for (int i = 0; i < T; i++) {
            As[buf][a_kk][ty + 16 * i] = ra[i];
            Bs[buf][b_kr + BR * i][b_col] = rb[i];
        }
    };

    double acc[T][T];
#pragma unroll
    for (int i = 0; i < T; i++)
#pragma unroll
        for (int j = 0; j < T; j++) acc[i][j] = 0.0;

    const int64_t ktiles = (k + BK - 1) / BK;
    if (ktiles > 0) {
        load_regs(0);
        store_smem(0);
        __syncthreads();
    }
    for (int64_t t = 0; t < ktiles; t++) {
        const int buf = (int)(t & 1);
        if (t + 1 < ktiles) load_regs((t + 1) * BK);
#pragma unroll
        for (int kk = 0; kk < BK; kk++) {
            double a[T], b[T];
#pragma unroll
            for (int i = 0; i < T; i++) a[i] = As[buf][kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < T; j++) b[j] = Bs[buf][kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < T; i++)
#pragma unroll
                for (int j = 0; j < T; j++) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        if (t + 1 < ktiles) {
            store_smem(buf ^ 1);
            __syncthreads();
        }
    }

#pragma unroll
    for (int i = 0; i < T; i++) {
        const int64_t r = m0 + ty + 16 * i;
        if (r >= m) continue;
#pragma unroll
        for (int j = 0; j < T; j++) {
            const int64_t c = n0 + tx + 16 * j;
            if (c >= n) continue;
            double v = alpha * acc[i][j];
            if (beta != 0.0) v = fma(beta, C[r * ldc + c], v);
            D[r * ldd + c] = v;
        }
    }
}

// An 8 x 16 or 8 x 8 output tile per CTA, one output per thread: products whose
// 16 x 16 tiles leave SMs idle (128^3 has 64 of them) or fill their last wave
// badly (256^3: 256 on 152 SMs).  A warp's chain of dependent FMAs (64 cycles
// each) is also all that an SM sub-partition's FP64 unit can take.  Same order
// of operations (k in order, zero padding to a multiple of BK) as the other
// tiles.
constexpr int SM_ROWS = 8;
template <int COLS>
__device__ __forceinline__ void gemm_f64_small_tile(int64_t m, int64_t n, int64_t k, double alpha,
                                                    const double* __restrict__ A, int64_t lda,
                                                    const double* __restrict__ B, int64_t ldb, double beta,
                                                    const double* C, int64_t ldc, double* D, int64_t ldd,
                                                    int64_t tile_m, int64_t tile_n) {
    constexpr int KS = 2 * BK;  // two k-steps per stage
    constexpr int THREADS = SM_ROWS * COLS, AR = THREADS / KS, AP = SM_ROWS / AR, BP = KS / SM_ROWS;
    __shared__ double As[2][KS][SM_ROWS + 1];
    __shared__ double Bs[2][KS][COLS];
    const int tid = threadIdx.x, tx = tid % COLS, ty = tid / COLS;
    const int64_t m0 = tile_m * SM_ROWS, n0 = tile_n * COLS;
    const int a_kk = tid % KS, a_r = tid / KS;  // A: AR rows per pass
    double ra[AP], rb[BP];
    auto load_regs = [&](int64_t k0) {
#pragma unroll
        for (int i = 0; i < AP; i++) {
            const int64_t r = m0 + a_r + AR * i, c = k0 + a_kk;
            ra[i] = (r < m && c < k) ? A[r * lda + c] : 0.0;
        }
#pragma unroll
        for (int i = 0; i < BP; i++) {
            const int64_t r = k0 + ty + SM_ROWS * i, c = n0 + tx;
            rb[i] = (r < k && c < n) ? B[r * ldb + c] : 0.0;
        }
    };
    auto store_smem = [&](int buf) {
#pragma unroll
        for (int i = 0; i < AP; i++) As[buf][a_kk][a_r + AR * i] = ra[i];
#pragma unroll
        for (int i = 0; i < BP; i++) Bs[buf][ty + SM_ROWS * i][tx] = rb[i];
    };
    double acc = 0.0;
    const int64_t kpad = (k + BK - 1) / BK * BK;
    if (kpad > 0) {
        load_regs(0);
        store_smem(0);
        __syncthreads();
    }
    for (int64_t k0 = 0, t = 0; k0 < kpad; k0 += KS, t++) {
        const int buf = (int)(t & 1);
        const bool more = k0 + KS < kpad;
        if (more) load_regs(k0 + KS);
#pragma unroll
        for (int kk = 0; kk < BK; kk++) acc = fma(As[buf][kk][ty], Bs[buf][kk][tx], acc);
        if (k0 + BK < kpad) {
#pragma unroll
            for (int kk = BK; kk < KS; kk++) acc = fma(As[buf][kk][ty], Bs[buf][kk][tx], acc);
        }
        if (more) {
            store_smem(buf ^ 1);
            __syncthreads();
        }
    }
    const int64_t r = m0 + ty, c = n0 + tx;
    if (r < m && c < n) {
        double v = alpha * acc;
        if (beta != 0.0) v = fma(beta, C[r * ldc + c], v);
        D[r * ldd + c] = v;
    }
}

// Output tile of this CTA.  With group > 1 consecutive CTAs walk `group`
// tile rows down before moving one tile column right, so that the CTAs
// resident at once cover a squarer block of the output and share more of
// their A row panels and B column panels in L2; group <= 1 is row-major
// order.  A bijection of the grid either way (the last group may be short).
__device__ __forceinline__ void tile_of(int group, int64_t& tile_m, int64_t& tile_n) {
    if (group <= 1) {
        tile_m = blockIdx.y;
        tile_n = blockIdx.x;
        return;
    }
    const int64_t gx = gridDim.x, gy = gridDim.y;
    const int64_t pid = (int64_t)blockIdx.y * gx + blockIdx.x;
    const int64_t per = (int64_t)group * gx;
    const int64_t g = pid / per, first = g * group;
    const int64_t rows = gy - first < group ? gy - first : (int64_t)group;
    const int64_t local = pid - g * per;
    tile_m = first + local % rows;
    tile_n = local / rows;
}

template <int TM>
__global__ void __launch_bounds__(NT, 2)
gemm_f64_kernel(int64_t m, int64_t n, int64_t k, double alpha, const double* __restrict__ A, int64_t lda,
                const double* __restrict__ B, int64_t ldb, double beta, const double* C, int64_t ldc,
                double* D, int64_t ldd, int group, const int* gate) {
    if (gate != nullptr && *gate == 0) return;
    int64_t tile_m, tile_n;
    tile_of(group, tile_m, tile_n);
    gemm_f64_tile<TM>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, D, ldd, tile_m, tile_n);
}

template <int COLS>
__global__ void __launch_bounds__(SM_ROWS * COLS)
gemm_f64_small_kernel(int64_t m, int64_t n, int64_t k, double alpha, const double* __restrict__ A, int64_t lda,
                      const double* __restrict__ B, int64_t ldb, double beta, const double* C, int64_t ldc, double* D,
                      int64_t ldd, const int* gate) {
    if (gate != nullptr && *gate == 0) return;
    gemm_f64_small_tile<COLS>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, D, ldd, blockIdx.y, blockIdx.x);
}

// Batched form: problem blockIdx.z uses the views described by the BatchView
// operands (same shape for every problem, per-problem base and leading dim).
template <int COLS>
__global__ void __launch_bounds__(SM_ROWS * COLS)
gemm_f64_small_batched_kernel(int64_t m, int64_t n, int64_t k, double alpha, BatchView a, BatchView b, double beta,
                              BatchView c, BatchView d) {
    const int z = blockIdx.z;
    const int64_t lda = a.ld_of(z), ldb = b.ld_of(z), ldd = d.ld_of(z);
    const int64_t ldc = beta != 0.0 ? c.ld_of(z) : 0;
    gemm_f64_small_tile<COLS>(m, n, k, alpha, a.ptr(z, lda), lda, b.ptr(z, ldb), ldb, beta,
                        beta != 0.0 ? c.ptr(z, ldc) : nullptr, ldc, const_cast<double*>(d.ptr(z, ldd)), ldd, blockIdx.y,
                        blockIdx.x);
}

template <int TM>
__global__ void __launch_bounds__(NT, 2)
gemm_f64_batched_kernel(int64_t m, int64_t n, int64_t k, double alpha, BatchView a, BatchView b, double beta,
                        BatchView c, BatchView d) {
    const int z = blockIdx.z;
    const int64_t lda = a.ld_of(z), ldb = b.ld_of(z), ldd = d.ld_of(z);
    const double* A = a.ptr(z, lda);
    const double* B = b.ptr(z, ldb);
    const double* C = nullptr;
    int64_t ldc = 0;
    if (beta != 0.0) {
        ldc = c.ld_of(z);
        C = c.ptr(z, ldc);
    }
    gemm_f64_tile<TM>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, const_cast<double*>(d.ptr(z, ldd)), ldd,
                      blockIdx.y, blockIdx.x);
}

// SPIN_F64_TILE=64|32|16 forces a tile size (for measurement); read once.
int forced_tile() {
    static int t = -1;
    if (t < 0) {
        const char* e = getenv("SPIN_F64_TILE");
        const int v = e ? atoi(e) : 0;
        t = (v == 64 || v == 32 || v == 16) ? v : 0;
    }
    return t;
}

// Tile rows per group of the single-product tile order (SPIN_F64_GROUP
// overrides it, for measurement; read once).
int tile_group() {
    static int g = -1;
    if (g < 0) {
        const char* e = getenv("SPIN_F64_GROUP");
        const int v = e ? atoi(e) : 0;
        g = v > 0 ? v : kTileGroup;
    }
    return g;
}

}  // namespace

int forced_f64_tile() { return forced_tile(); }

// Tile for an m x n product (count of them side by side): the one whose
// busiest SM has the fewest FMAs, ceil(tiles / 152) * rows * cols per k, larger
// tiles preferred unless a smaller one has 1 % fewer: all of them keep the FP64
// pipe equally busy, so that count is the time (within 3 % of ceil(tiles / 152)
// rows cols k / (2 per clock) plus 4 us).  us with 64, 32, 16 rows, 8 x 16 and
// 8 x 8: 128^3 -, 35.6, 11.1, 7.6, 7.4; 200^3 -, 56.4, 29.1, 21.9, 18.9; 256^3
// -, 69.1, 35.3, 34.4, 30.7; 300^3 -, 81.7, 60.5, 50.1, 50.6; 512^3 -, 257.9,
// 229.2, 228.6, 229.6; 1024^3 2046, 1791, 1736, 1740, 1748 (at 64 rows until a
// smaller tile was 25 % better, 512^3 took 258 and 1024^3 2046).
F64Tile gemm_f64_tile_size(int64_t m, int64_t n, int64_t count) {
    const int forced = forced_tile();
    if (forced) return {forced, forced};
    constexpr F64Tile tiles[] = {{64, 64}, {32, 32}, {16, 16}, {8, 16}, {8, 8}};
    F64Tile best = tiles[0];
    double best_cost = 0.0;
    for (const F64Tile& t : tiles) {
        const int64_t rows = (m + t.rows - 1) / t.rows;
        const double num = (double)rows * (double)((n + t.cols - 1) / t.cols) * (double)count;
        const double cost = std::ceil(num / 152.0) * t.rows * t.cols;
        if (t.rows == 64 || (rows <= 65535 && cost * 1.01 <= best_cost)) {  // blockIdx.y
            best = t;
            best_cost = cost;
        }
    }
    return best;
}

int launch_gemm_f64_batched(int64_t m, int64_t n, int64_t k, double alpha, const BatchView& a, const BatchView& b,
                            double beta, const BatchView& c, const BatchView& d, int count, cudaStream_t s) {
    if (m <= 0 || n <= 0 || count <= 0) return SPIN_OK;
    const F64Tile t = gemm_f64_tile_size(m, n, count);
    const dim3 grid((unsigned)((n + t.cols - 1) / t.cols), (unsigned)((m + t.rows - 1) / t.rows), (unsigned)count);
    if (grid.y > 65535u || grid.z > 65535u) return SPIN_ERR_INVALID_ARG;
    auto kernel = t.rows == 64   ? gemm_f64_batched_kernel<64>
                  : t.rows == 32 ? gemm_f64_batched_kernel<32>
                  : t.rows == 16 ? gemm_f64_batched_kernel<16>
                  : t.cols == 16 ? gemm_f64_small_batched_kernel<16>
                                 : gemm_f64_small_batched_kernel<8>;
    kernel<<<grid, t.rows >= 16 ? NT : t.rows * t.cols, 0, s>>>(m, n, k, alpha, a, b, beta, c, d);
    SPIN_CUDA_TRY(cudaGetLastError());
    return SPIN_OK;
}

int launch_gemm_f64(int64_t m, int64_t n, int64_t k, double alpha, const double* A, int64_t lda,
                    const double* B, int64_t ldb, double beta, const double* C, int64_t ldc, double* D,
                    int64_t ldd, cudaStream_t s, const int* gate) {
    if (m <= 0 || n <= 0) return SPIN_OK;
    const F64Tile t = gemm_f64_tile_size(m, n, 1);
    const dim3 grid((unsigned)((n + t.cols - 1) / t.cols), (unsigned)((m + t.rows - 1) / t.rows));
    if (grid.y > 65535u) return SPIN_ERR_INVALID_ARG;
    if (t.rows < 16) {
        auto kernel = t.cols == 16 ? gemm_f64_small_kernel<16> : gemm_f64_small_kernel<8>;
        kernel<<<grid, t.rows * t.cols, 0, s>>>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, D, ldd, gate);
    } else {
        auto kernel = t.rows == 64 ? gemm_f64_kernel<64> : t.rows == 32 ? gemm_f64_kernel<32> : gemm_f64_kernel<16>;
        kernel<<<grid, NT, 0, s>>>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, D, ldd, tile_group(), gate);
    }
    SPIN_CUDA_TRY(cudaGetLastError());
    return SPIN_OK;
}

}  // namespace spin
