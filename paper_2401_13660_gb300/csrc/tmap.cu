// What the launchers share on the host: TMA tensor-map encoding, device limits. cuTensorMapEncodeTiled is
// fetched through the runtime's driver entry point, so the library does not
// link libcuda directly.
#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>
#include <mutex>

#include "internal.h"

namespace mbscan {
namespace {

using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                   const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                   const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault,
                                             &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<EncodeTiledFn>(f);
    }();
    return fn;
}

}  // namespace

bool encode_tmap(CUtensorMap *m, const void *base, int elem_bytes, int rank, const uint64_t *dims,
                 const uint64_t *strides, const uint32_t *box, int swizzle) {
    if (swizzle != 0 && swizzle != 64 && swizzle != 128) return false;
    EncodeTiledFn enc = encode_fn();
    if (!enc || rank < 1 || rank > 5) return false;
    cuuint64_t d[5], st[4];
    cuuint32_t bx[5], es[5];
    for (int i = 0; i < rank; ++i) {
        d[i] = dims[i];
        bx[i] = box[i];
        es[i] = 1;
        if (i + 1 < rank) st[i] = strides[i];
    }
    const CUtensorMapDataType dt = elem_bytes == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                   : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    return enc(m, dt, (cuuint32_t)rank, const_cast<void *>(base), d, st, bx, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE,
               swizzle == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                              : (swizzle == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE),
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

const DeviceLimits *device_limits() {
    constexpr int kMaxDevices = 64;
    static DeviceLimits lim[kMaxDevices];
    static std::atomic<int> ready[kMaxDevices];   // 0: not read yet, 1: lim[] is filled
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    if (!ready[dev].load(std::memory_order_acquire)) {
        std::lock_guard<std::mutex> guard(mu);
        if (!ready[dev].load(std::memory_order_relaxed)) {
            int v[4];
            const cudaDeviceAttr attr[4] = {cudaDevAttrMultiProcessorCount, cudaDevAttrMaxSharedMemoryPerMultiprocessor,
                                            cudaDevAttrReservedSharedMemoryPerBlock,
                                            cudaDevAttrMaxSharedMemoryPerBlockOptin};
            for (int i = 0; i < 4; ++i)
                if (cudaDeviceGetAttribute(&v[i], attr[i], dev) != cudaSuccess) return nullptr;
            if (v[0] <= 0) return nullptr;
            lim[dev] = DeviceLimits{v[0], (size_t)v[1], (size_t)v[2], (size_t)v[3]};
            ready[dev].store(1, std::memory_order_release);
        }
    }
    return &lim[dev];
}

int device_sms() {
    const DeviceLimits *l = device_limits();
    return l ? l->sms : 0;
}

size_t spread_smem(size_t smem, int64_t grid, int per) {
    const DeviceLimits *l = device_limits();
    if (!l) return smem;
    const int64_t m = (grid + l->sms - 1) / l->sms;
    if (m >= per) return smem;
    const size_t want = l->smem_sm / (size_t)(m + 1) - l->smem_reserved + 128;   // m of these fit, m + 1 do not
    return want > smem && want <= l->smem_optin ? want : smem;
}

Placement place_scan(int64_t L, int64_t grid, int per, size_t smem) {
    const int64_t sms = device_sms();
    if (L < 256 || grid > (per - 1) * sms) return {true, smem};
    if (grid <= sms) return {false, smem};
    return {true, spread_smem(smem, grid, per)};
}

}  // namespace mbscan
