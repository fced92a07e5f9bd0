// Kernel launchers (host functions defined next to their kernels).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/comet.h"
#include "params.h"

namespace comet {

// A launch that may begin while the kernel before it in the stream still runs (programmatic
// dependent launch): its blocks set up and then wait in pdl_wait() for that kernel's end.  Every
// kernel launched this way calls pdl_wait() in every thread before it touches memory that another
// kernel reads or writes.  A kernel calls pdl_launch() near its end, not at its start: the next
// grid's blocks would otherwise take whatever room this one leaves and stay unevenly spread over the
// SMs (a 256-tile grid of k_gemm_small.cu took 21 us instead of 16).  Only the pre-passes call it
// early: the next one is the other operand's, or a GEMM with one block per SM.
template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A &&...args) {
    cudaLaunchConfig_t c = {};
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a[0].val.programmaticStreamSerializationAllowed = 1;
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = a;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

#if defined(__CUDACC__)
// Waits for the end (and the memory) of the kernel before this one; nothing when it has ended
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel of the stream begin once every block has come here (or ended)
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

// One operand of the abs-max kernel: dense (n elements) or a view (r, strides s0)
struct AbsmaxArg {
    const void *x;
    int64_t n;
    Radix r;
    int view;
    uint32_t blocks;               // blocks given to the operand = slots it fills
    void *slots;                   // 8-byte words, one per block: the bits of its largest |x|
};

// Blocks (and slots) the abs-max of n elements uses, at most `room`
uint32_t absmax_blocks(int64_t n, int elem_bytes, uint32_t room);

// The largest finite |x| of one or two operands (b.blocks = 0: one), in one launch, into their slots
cudaError_t launch_absmax(const AbsmaxArg &a, const AbsmaxArg &b, int elem_bytes, cudaStream_t s);

cudaError_t launch_move(const XposeParams &p, int elem_bytes, int vi, int vo, cudaStream_t s);
cudaError_t launch_scale(const XposeParams &p, int elem_bytes, int vi, int vo, cudaStream_t s);
cudaError_t launch_split(const XposeParams &p, int elem_bytes, int vi, int vo, cudaStream_t s);
cudaError_t launch_split6(const XposeParams &p, int elem_bytes, int vi, int vo, cudaStream_t s);

cudaError_t launch_gemm_f64(const GemmParams &p, int elem_bytes, bool a_kcontig, bool b_kcontig,
                            cudaStream_t s);

// small FP32 GEMMs in one launch (k_gemm_small.cu)
cudaError_t launch_gemm_small(const GemmParams &p, bool a_kcontig, bool b_kcontig, cudaStream_t s);

cudaError_t launch_fill(void *out, int64_t n, double value, int elem_bytes, cudaStream_t s);

// Two FP16 planes per operand.  want_ksplit: 0 = K slices and tile width by split_schedule, k = k
// slices; kc: upper limit of a chunk's K values (0 = none); FP32 partials of the slices in `partial` (as many as fit partial_bytes), summed by a
// reduce kernel into C.
cudaError_t launch_gemm_split(const GemmParams &p, const void *parts_a, const void *parts_b,
                              int64_t kpad, const void *scale_a, const void *scale_b,
                              int64_t kc, int out_bytes, int debug_flags, cudaStream_t s,
                              uint32_t want_ksplit, float *partial, int64_t partial_bytes);

// `partial`: room for the int64 sums of K slices (emu_schedule; as many as fit partial_bytes)
cudaError_t launch_gemm_emu(const GemmParams &p, const void *parts_a, const void *parts_b, int64_t kpad,
                            const void *scale_a, const void *scale_b, int debug_flags, cudaStream_t s,
                            long long *partial, int64_t partial_bytes);

cudaError_t launch_gemv(const GemvParams &p, int elem_bytes, cudaStream_t s);

// device status word of the current device (set by kernels whose waits run out)
int *device_status_word();

}  // namespace comet
