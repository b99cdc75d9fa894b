// Pieces that the tensor-core product kernels share (tc_gemm.cu, crt.cu):
// tile and ring sizes, the control block in shared memory, output views, the
// sources that the operand splits read, row and column exponents, tensor maps.
#pragma once
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "common.cuh"
#include "tc_gemm.h"
#include "tc_ptx.cuh"

namespace spin {
namespace {

using namespace tc;

constexpr int BM = 128, BK = 64;
constexpr int GROUP_M = 8;  // row blocks per rasterisation band
constexpr uint32_t A_TILE_BYTES = BM * BK * 2;  // 16 KB
constexpr uint64_t WAIT_LIMIT_NS = 10ull * 1000 * 1000 * 1000;
constexpr int STAGES_MAX = 8;

template <int BN, int KS>
struct Cfg {
    static constexpr uint32_t B_TILE_BYTES = BN * BK * 2;
    static constexpr uint32_t STAGE_BYTES = KS * (A_TILE_BYTES + B_TILE_BYTES);
    static constexpr int STAGES = (196608 / STAGE_BYTES) > 6 ? 6 : (196608 / STAGE_BYTES);  // ~192 KB ring
    static constexpr uint32_t TMEM_COLS = 2 * BN <= 256 ? 256 : 512;  // power of two >= 2 BN
    static constexpr size_t SMEM_BYTES = 1024 /*align slack*/ + STAGES * STAGE_BYTES + 256 /*barriers etc.*/;
};

struct SmemCtl {
    uint64_t full[STAGES_MAX];
    uint64_t empty[STAGES_MAX];
    uint64_t tfull[2];
    uint64_t tempty[2];
    uint64_t final_bar;
    uint32_t tmem_base;
    int abort;
    int issued;  // pair kernel: stage uses this CTA's producer issued
};
static_assert(sizeof(SmemCtl) <= 256, "control block");

__device__ __forceinline__ void raise_timeout(SmemCtl* ctl, int* err) {
    ctl->abort = 1;
    if (err) atomicCAS(err, 0, SPIN_ERR_TIMEOUT);
}

template <int EPI_WARPS>
struct Epi {
    static constexpr int THREADS = 64 + 32 * EPI_WARPS;
    // registers are granted per group of four warps: budget for the rounded-up count
    static constexpr int ALLOC_THREADS = (THREADS + 127) / 128 * 128;
    static constexpr int MAXREG = (65536 / ALLOC_THREADS) / 8 * 8 > 255 ? 248 : (65536 / ALLOC_THREADS) / 8 * 8;
};

// Row grow of D (and of C, or null) for problem z.
__device__ __forceinline__ double* out_row(const TcGemmParams& p, int z, int grow) {
    if (!p.batch) return p.D + (int64_t)grow * p.ldd;
    const int64_t ld = p.d_lds ? p.d_lds[z] : p.d_ld;
    return p.d_base[z] + (p.d_r0 + grow) * ld + p.d_c0;
}
__device__ __forceinline__ const double* in_row(const TcGemmParams& p, int z, int grow) {
    if (!p.batch) return p.C ? p.C + (int64_t)grow * p.ldc : nullptr;
    if (!p.c_base) return nullptr;
    const int64_t ld = p.c_lds ? p.c_lds[z] : p.c_ld;
    return p.c_base[z] + (p.c_r0 + grow) * ld + p.c_c0;
}

// Operand source of a split: one FP64 view, or problem z's view of a batch.
// act (optional): problem z is split only while act[z] != 0.  nv
// (optional): the sum of squares of problem z covers only its leading
// nv[z] x nv[z] block (a matrix padded with the identity).
struct SrcOne {
    const double* p;
    int64_t ld;
    const int* act;
    __device__ __forceinline__ const double* row(int, int r) const { return p + (int64_t)r * ld; }
    __device__ __forceinline__ bool on(int) const { return act == nullptr || act[0] != 0; }
    __device__ __forceinline__ int valid(int) const { return 0x7fffffff; }
};
struct SrcMany {
    BatchView v;
    const int* act;
    const int* nv;
    __device__ __forceinline__ const double* row(int z, int r) const {
        const int64_t l = v.ld_of(z);
        return v.base[z] + (v.r0 + r) * l + v.c0;
    }
    __device__ __forceinline__ bool on(int z) const { return act == nullptr || act[z] != 0; }
    __device__ __forceinline__ int valid(int z) const { return nv ? nv[z] : 0x7fffffff; }
};

__device__ __forceinline__ uint16_t bf16_bits(float f) {
    return __bfloat16_as_ushort(__float2bfloat16_rn(f));
}

// ---------------------------------------------- row and column exponents --

// Biased exponent field of x (0 for zero and subnormals).  The exponent e
// with max|x| < 2^e (frexp convention) of a row is max(field) - 1022: the
// largest magnitude has the largest field.  Integer work only.
__device__ __forceinline__ int exp_field(double x) {
    return (int)((unsigned long long)__double_as_longlong(x) >> 52) & 0x7FF;
}

// Per-row max exponent of an FP64 matrix (one warp per row) and optional
// sum of squares of all entries.
template <class Src>
__global__ void row_exp_kernel(Src src, int rows, int cols, int* __restrict__ ex, int64_t exs, double* sumsq,
                               int64_t sss) {
    const int z = blockIdx.z;
    if (!src.on(z)) return;
    const int warps = blockDim.x >> 5;
    const int r = blockIdx.x * warps + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (r >= rows) return;
    const double* sr = src.row(z, r);
    const int nv = src.valid(z);
    const bool sum_row = sumsq != nullptr && r < nv;
    int m = 0;
    double ss = 0.0;
    for (int c = lane; c < cols; c += 32) {
        const double v = sr[c];
        m = max(m, exp_field(v));
        if (sum_row && c < nv) ss = fma(v, v, ss);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        m = max(m, __shfl_down_sync(0xffffffffu, m, off));
        ss += __shfl_down_sync(0xffffffffu, ss, off);
    }
    if (lane == 0) {
        ex[z * exs + r] = m - 1022;
        if (sumsq) atomicAdd(sumsq + z * sss, ss);
    }
}

// Per-column max exponent: atomicMax of exponent fields on a zero start,
// converted to the frexp convention by col_exp_finish_kernel.
template <class Src>
__global__ void col_exp_kernel(Src src, int rows, int cols, int rows_per_block, int* __restrict__ ex, int64_t exs,
                               double* sumsq, int64_t sss) {
    const int z = blockIdx.z;
    if (!src.on(z)) return;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int r0 = blockIdx.y * rows_per_block;
    const int r1 = min(rows, r0 + rows_per_block);
    int m = 0;
    const int nv = src.valid(z);
    const bool sum_col = sumsq != nullptr && c < nv;
    double ss4[4] = {0.0, 0.0, 0.0, 0.0};  // four FMA chains: a dependent FP64 FMA takes 64+ cycles here
    if (c < cols) {
        int r = r0;
        for (; r + 3 < r1; r += 4) {
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const double v = src.row(z, r + u)[c];
                m = max(m, exp_field(v));
                if (sum_col && r + u < nv) ss4[u] = fma(v, v, ss4[u]);
            }
        }
        for (; r < r1; r++) {
            const double v = src.row(z, r)[c];
            m = max(m, exp_field(v));
            if (sum_col && r < nv) ss4[0] = fma(v, v, ss4[0]);
        }
    }
    double ss = (ss4[0] + ss4[1]) + (ss4[2] + ss4[3]);
    if (c < cols && m > 0) atomicMax(&ex[z * exs + c], m);
    if (sumsq) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) ss += __shfl_down_sync(0xffffffffu, ss, off);
        if ((threadIdx.x & 31) == 0 && ss != 0.0) atomicAdd(sumsq + z * sss, ss);
    }
}

__global__ void col_exp_finish_kernel(int* ex, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) ex[i] -= 1022;
}

__global__ void fill_int_kernel(int* p, int64_t n, int v) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}

// Grid of a row-wise split: blocks per problem so that the whole launch has
// about 16 blocks per SM.
inline dim3 rows_grid(int64_t total, int count) {
    const int64_t per = std::max<int64_t>(1, (152 * 16) / std::max(1, count));
    return dim3((unsigned)std::min<int64_t>((total + 255) / 256, per), 1, (unsigned)count);
}

// Exponents of every row (transpose: of every column) of `count` problems,
// and the sums of squares (optional); 1 or 3 launches.
template <class Src>
int operand_exponents(Src src, int rows, int cols, bool transpose, int* ex, double* sumsq, int64_t sss, int count,
                      cudaStream_t s) {
    if (!transpose) {
        row_exp_kernel<Src><<<dim3((unsigned)((rows + 7) / 8), 1, (unsigned)count), 256, 0, s>>>(
            src, rows, cols, ex, rows, sumsq, sss);
    } else {
        const int64_t nex = (int64_t)cols * count;
        fill_int_kernel<<<(unsigned)((nex + 255) / 256), 256, 0, s>>>(ex, nex, 0);
        // rows per block: enough blocks to cover the SMs at small orders,
        // at most 256 (fewer atomics at large ones)
        const int64_t col_blocks = (int64_t)((cols + 255) / 256) * count;
        int rpb = (int)std::min<int64_t>(256, std::max<int64_t>(16, (int64_t)rows * col_blocks / 608));
        rpb = (rpb + 7) & ~7;
        const dim3 g1((unsigned)((cols + 255) / 256), (unsigned)((rows + rpb - 1) / rpb), (unsigned)count);
        col_exp_kernel<Src><<<g1, 256, 0, s>>>(src, rows, cols, rpb, ex, cols, sumsq, sss);
        col_exp_finish_kernel<<<(unsigned)((nex + 255) / 256), 256, 0, s>>>(ex, nex);
    }
    SPIN_CUDA_TRY(cudaGetLastError());
    return SPIN_OK;
}

// ----------------------------------------------------------- tensor maps --

inline PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (fn == nullptr) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

inline int make_map(CUtensorMap* m, const uint16_t* base, int64_t inner, int64_t outer, int64_t ld_elems, uint32_t box_rows) {
    auto fn = encode_fn();
    if (fn == nullptr) return SPIN_ERR_CUDA;
    if (((uintptr_t)base & 15u) != 0 || (ld_elems * 2) % 16 != 0) return SPIN_ERR_INVALID_ARG;
    cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
    cuuint64_t strides[1] = {(cuuint64_t)(ld_elems * 2)};
    cuuint32_t box[2] = {(cuuint32_t)BK, box_rows};
    cuuint32_t es[2] = {1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)base, dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? SPIN_OK : SPIN_ERR_CUDA;
}

inline int sm_count() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return 152;
    }
    return n > 0 ? n : 152;
}

}  // namespace
}  // namespace spin
