// Small device helpers shared by the convolution kernels.
#ifndef RTOSS_CONV_COMMON_CUH
#define RTOSS_CONV_COMMON_CUH

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <atomic>

#include "rtoss_internal.h"

namespace rtoss_dev {

template <typename T> __device__ __forceinline__ float to_f32(T v);
template <> __device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <> __device__ __forceinline__ float to_f32<__half>(__half v) { return __half2float(v); }

template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
template <> __device__ __forceinline__ __half from_f32<__half>(float v) { return __float2half_rn(v); }

// Packed value i of the given storage type, widened to fp32.
__device__ __forceinline__ float load_val(const void* val, size_t i, int dtype) {
    if (dtype == RTOSS_F32) return reinterpret_cast<const float*>(val)[i];
    if (dtype == RTOSS_BF16) return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(val)[i]);
    return __half2float(reinterpret_cast<const __half*>(val)[i]);
}

// The same for kernels that read a handle ahead of their wait (see pdl_enter).
__device__ __forceinline__ float load_val_cg(const void* val, size_t i, int dtype) {
    if (dtype == RTOSS_F32) return __ldcg(reinterpret_cast<const float*>(val) + i);
    const unsigned short bits = __ldcg(reinterpret_cast<const unsigned short*>(val) + i);
    return dtype == RTOSS_BF16 ? __bfloat162float(__ushort_as_bfloat16(bits)) : __half2float(__ushort_as_half(bits));
}

// The k values of kernel kid, in as few loads as their size allows (kernels start on multiples of it).
__device__ __forceinline__ void load_vals_cg(const void* val, size_t kid, int k, int dtype, float (&v)[9]) {
    const int bytes = k * (dtype == RTOSS_F32 ? 4 : 2);
    unsigned u[4] = {0u, 0u, 0u, 0u};
    if (bytes == 16) {
        const uint4 q = __ldcg(reinterpret_cast<const uint4*>(val) + kid);
        u[0] = q.x, u[1] = q.y, u[2] = q.z, u[3] = q.w;
    } else if (bytes == 8) {
        const uint2 q = __ldcg(reinterpret_cast<const uint2*>(val) + kid);
        u[0] = q.x, u[1] = q.y;
    } else {
#pragma unroll
        for (int j = 0; j < 9; ++j) v[j] = j < k ? load_val_cg(val, kid * k + j, dtype) : 0.f;
        return;
    }
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        if (dtype == RTOSS_F32) {
            v[j] = j < 4 ? __uint_as_float(u[j & 3]) : 0.f;
        } else {
            const unsigned short h = j < 8 ? (unsigned short)(u[(j >> 1) & 3] >> (16 * (j & 1))) : (unsigned short)0;
            v[j] = dtype == RTOSS_BF16 ? __bfloat162float(__ushort_as_bfloat16(h)) : __half2float(__ushort_as_half(h));
        }
    }
}

// Fused epilogue: bias was already added by the caller; activation in fp32.
__device__ __forceinline__ float activate(float v, int act) {
    if (act == RTOSS_ACT_RELU) return fmaxf(v, 0.f);
    if (act == RTOSS_ACT_SILU) return v / (1.f + __expf(-v));
    return v;
}

// Programmatic dependent launch.  Every kernel of the library is launched with programmatic stream serialization: it lets
// the NEXT kernel of the stream be scheduled already (launch latency and block start-up then overlap this kernel's run),
// and waits until every kernel before it in the stream has completed and its writes are visible before it touches memory
// that those may write or still read.  Most kernels do both at once, in pdl_enter().
//
// One kind of memory is read ahead of the wait: a packed handle's arrays (values, ids, masks, the tensor path's weights and
// issue words) by the convolutions (conv_tc_kernel, conv_few_kernel, conv3x3_stem_mma_kernel) and by to_dense_kernel, and a
// batch's own tables by the ordering kernel.  They are constant while a network runs.  What makes it sound:
//   - the kernels that WRITE a handle begin with pdl_enter_handle_writer(): they wait like every other kernel but do not let
//     the next one start, so a reader starts after the writer has completed.  (One exception: the first kernel of the
//     whole-model pass lets the ordering kernel behind it start early, which is a writer itself: it waits for the first
//     kernel's end before it reads an id and lets nothing start before its own.)
//   - they end with handle_writer_done(): whatever they wrote is performed before the block leaves;
//   - the readers take it from L2 (__ldcg, bulk copies): without an acquire of their own nothing orders this SM's L1 behind
//     the writer.  Where many CTAs read the same few lines that way, a CTA asks for each line once, or the loads queue up.
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ void pdl_enter_handle_writer() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// (All threads of the block: the barrier hands their writes to the thread whose fence then covers them all.)
__device__ __forceinline__ void handle_writer_done() {
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("fence.acq_rel.gpu;" ::: "memory");
}

// The kernels that write handles follow one another in pairs whose shared memory differs (6 to 46 KB a block).  An SM that has
// to move the line between its shared memory and its L1 first runs empty, which cost 5 us between two of them: all of them
// ask for the same line (a hint; set once per device, before a kernel's first launch).
template <auto kKernel>
inline void writers_carveout() {
    static std::atomic<bool> done[64];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || done[dev].load(std::memory_order_relaxed)) return;
    if (cudaFuncSetAttribute(kKernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) != cudaSuccess) cudaGetLastError();
    done[dev].store(true, std::memory_order_relaxed);
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                              Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<Args&&>(args)...);
}

// The same with thread-block clusters of `cluster` CTAs along x (1 = no clusters).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, int cluster,
                              Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<Args&&>(args)...);
}

}  // namespace rtoss_dev

#endif
