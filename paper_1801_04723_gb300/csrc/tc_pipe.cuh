// Pieces that the tensor-core product kernels share (tc_gemm.cu, crt.cu):
// tile and ring sizes, the control block in shared memory, output views,
// tensor maps.
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
