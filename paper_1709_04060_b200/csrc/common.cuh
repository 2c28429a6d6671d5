// Shared host-side helpers of the qnn C ABI implementation (sm_100a only).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

#include <atomic>

#include "qnn.h"

namespace qnn {

// Host counter of kernels launched by this library (reported by benchmarks).
extern std::atomic<unsigned long long> g_launches;

inline void count_launch(int n = 1) { g_launches.fetch_add((unsigned long long)n, std::memory_order_relaxed); }

// Per-device host caches are arrays of this size; a device index beyond it is an error.
constexpr int QNN_MAX_DEVICES = 64;

// Index of the current device, or -1 (CUDA error, or an index the caches cannot hold).
inline int current_device() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= QNN_MAX_DEVICES) return -1;
    return dev;
}

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline bool aligned4(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 3u) == 0; }     // thresholds (or none)

inline int round_up(int x, int m) { return (x + m - 1) / m * m; }
inline int ceil_div(int x, int m) { return (x + m - 1) / m; }

inline bool valid_enc(int enc, int bits) {
    if (enc == QNN_ENC_BIPOLAR) return bits == 1;
    return enc == QNN_ENC_UNSIGNED || enc == QNN_ENC_SIGNED;
}

inline qnn_status launch_status() {
    return cudaGetLastError() == cudaSuccess ? QNN_OK : QNN_ERR_CUDA;
}

// Programmatic dependent launch.  The tensor-core GEMMs, the few-column kernels and small pools are
// launched so that their CTAs may be placed while the previous kernel of the stream drains (they
// wait in griddepcontrol.wait before touching global memory).  The other kernels only do their part
// as predecessors: pdl_trigger() tells the scheduler that a dependent may start placing CTAs (no
// effect unless the next kernel asked for it), pdl_wait() is a no-op for a normally launched
// kernel.  They are not launched that way themselves: early placement next to a draining kernel
// packs the CTAs of a small grid onto few SMs, which halved the bit-serial kernel's speed.
// A kernel launched this way is resident while the one ahead may still write what it will read, so it
// reads global memory with plain loads only: ld.global.nc (__ldg, const __restrict__) is for data that
// nothing writes as long as the kernel lives.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_enter() {
    pdl_trigger();
    pdl_wait();
}
// A plain load that the compiler may issue ahead of stores to shared memory around it, which an ordinary access may
// not be (it could alias them), but not ahead of pdl_wait() (volatile statements keep their order).  Thresholds
// staged by ordinary loads: up to 7 % longer in a kernel bound by its epilogue (263 x 263 -> 48, 1 x 1, batch 26: 195 ->
// 208 us).
__device__ __forceinline__ int32_t ld_global(const int32_t *p) {
    int32_t v;
    asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ld_global(const uint32_t *p) { return (uint32_t)ld_global(reinterpret_cast<const int32_t *>(p)); }
__device__ __forceinline__ uint4 ld_global(const uint4 *p) {
    uint4 v;
    asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
#endif

#ifdef __CUDACC__
// Lets a kernel be launched with up to `limit` bytes of dynamic shared memory.  The attribute is set once
// per kernel and device (`done`: static, one flag per device), always to the same limit: threads that
// arrive here together write the same number, so no order of theirs leaves an attribute below what a
// launch needs (one that followed the largest size seen so far could be lowered by a second thread).
constexpr size_t SMEM_LIMIT = 227 * 1024;
template <typename Kernel>
inline bool allow_smem(Kernel *kern, size_t limit, std::atomic<bool> &done) {
    if (done.load(std::memory_order_relaxed)) return true;
    if (cudaFuncSetAttribute(reinterpret_cast<const void *>(kern), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit) != cudaSuccess)
        return false;
    done.store(true, std::memory_order_relaxed);
    return true;
}

// Launch with programmatic stream serialization (see above): the launch gap overlaps the tail of the
// kernel ahead.  For kernels that wait in griddepcontrol.wait before they touch global memory.
template <typename Params>
inline cudaError_t launch_pdl(void (*kern)(const Params), dim3 grid, int threads, size_t smem, cudaStream_t s, const Params &p) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3((unsigned)threads); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, p);
}
#endif

// Number of SMs of the current device (cached per device).
int sm_count();

// Path implementations (one translation unit each).
qnn_status pack_launch(const qnn_pack_desc *d, const void *logical, void *packed, cudaStream_t s);
qnn_status planes_to_int8_launch(const qnn_pack_desc *d, const void *planes, void *packed, cudaStream_t s,
                                 const qnn_pack_desc *d2 = nullptr, const void *planes2 = nullptr, void *packed2 = nullptr);
qnn_status gemm_bitserial_launch(const qnn_gemm_desc *d, const void *W, const void *A,
                                 const int32_t *thr, void *out, cudaStream_t s);
qnn_status gemm_bitserial_conv_launch(const qnn_conv_desc *cv, const qnn_gemm_desc *g, const void *W,
                                      const void *in, const int32_t *thr, void *out, cudaStream_t s);
bool gemv_mma_takes(const qnn_gemm_desc *d, bool has_thr);
qnn_status gemv_mma_launch(const qnn_gemm_desc *d, const void *W, const void *A,
                           const int32_t *thr, void *out, cudaStream_t s);
bool gemv_i8_fits(const qnn_gemm_desc *d);
qnn_status gemv_i8_launch(const qnn_gemm_desc *d, const void *W, const void *A,
                          const int32_t *thr, void *out, cudaStream_t s);
bool gemv_planes_fits(const qnn_gemm_desc *d);
qnn_status gemv_planes_launch(const qnn_gemm_desc *d, const void *W, const void *A,
                              const int32_t *thr, void *out, cudaStream_t s);
bool gemv_fields_dp4a_fits(const qnn_gemm_desc *d);
qnn_status gemv_fields_dp4a_launch(const qnn_gemm_desc *d, const void *W, const void *A,
                                   const int32_t *thr, void *out, cudaStream_t s);
bool gemv_fields_fits(const qnn_gemm_desc *d, bool has_thr);
qnn_status gemv_fields_launch(const qnn_gemm_desc *d, const void *W, const void *A,
                              const int32_t *thr, void *out, cudaStream_t s);
qnn_status gemm_tc_launch(const qnn_gemm_desc *d, const void *W, const void *A,
                          const int32_t *thr, void *out, void *ws, size_t ws_bytes, cudaStream_t s);
size_t gemm_tc_workspace_bytes(const qnn_gemm_desc *d);   // optional scratch of the CTA-pair kernel (0: none)
bool gemm_tc_uses_pair_kernel(const qnn_gemm_desc *d);
qnn_status gemm_tc_conv_launch(const qnn_conv_desc *cv, const qnn_gemm_desc *g, const void *W, const void *in,
                               const int32_t *thr, void *out, bool any_size, cudaStream_t s);
bool gemm_tc_conv_takes(const qnn_conv_desc *cv);       // what the tensor-map loader can lower
int gemm_tc_conv_boxes(const qnn_conv_desc *cv, const qnn_gemm_desc *g, bool has_thr, int *w, int *h, int *n);
qnn_status gemm_tc_lower_launch(const qnn_conv_desc *cv, const qnn_gemm_desc *g, const void *W, const void *in,
                                const int32_t *thr, void *out, cudaStream_t s);
qnn_status gemm_tc_planes_launch(const qnn_conv_desc *cv, const qnn_gemm_desc *g, const void *W, const void *A,
                                 const int32_t *thr, void *out, cudaStream_t s);
bool conv_direct_takes(const qnn_conv_desc *cv, const qnn_gemm_desc *g, bool has_thr, bool pool);
qnn_status conv_direct_launch(const qnn_conv_desc *cv, const qnn_gemm_desc *g, const void *W, const void *in,
                              const int32_t *thr, void *out, bool pool, cudaStream_t s);
qnn_status im2col_launch(const qnn_conv_desc *d, const void *in, void *lowered, cudaStream_t s);
qnn_status maxpool_launch(const qnn_pool_desc *d, const void *in, void *out, cudaStream_t s);
qnn_status validate_thresholds_launch(const int32_t *thr, int M, int n_thr, int *n_bad, cudaStream_t s);
qnn_status device_status_read(int *status);

}  // namespace qnn
