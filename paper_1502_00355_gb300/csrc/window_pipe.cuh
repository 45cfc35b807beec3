// window_pipe.cuh -- what the pass kernels share in working through a window
// stream (window.cuh): list entries, asynchronous copies, the slots in which
// headers and idle marks are held ahead of their use.
#pragma once

#include "device.cuh"
#include "window.cuh"

namespace sls {

// A block keeps two windows in shared memory: the one it works on and the
// next one, which is copied in meanwhile.  Headers are fetched three windows
// ahead and halo ids two, because each names what the next copies.
struct __align__(16) Ahead {
    uint32_t hdr[4][win::kHeaderWords];  // window i's header in slot i & 3
    uint8_t idle[4][4];                  // skip_unchanged: its subtiles that need no work
};

// Asynchronous copies global -> shared (no registers held while they fly).
__device__ __forceinline__ void copy16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy8(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy4(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ---- launches that overlap the one before -----------------------------------
// A pass kernel may be made resident while the kernel before it in its stream
// still runs (launch_early): the windows' headers and halo ids, which no pass
// writes, are fetched in the meantime, into the slots of blocks that have
// ended.  Everything a pass writes (coordinates, statistics) is touched only
// after after_previous(), which returns when the kernels before are complete
// and their writes visible; only then may the next kernel start early too, so
// at most two passes are resident at a time.  A launch costs a pass the
// emptying of the chip, the launch and two latencies of L2 in a row
// otherwise: per call, 100 passes of 1024^2 nodes 6.03 -> 5.92 ms, 38 Form B
// sweeps (seven launches each) of 1500 x 1100 7.68 -> 6.47 ms, 50 binary32
// passes of 2048^2 6.40 -> 6.17 ms.
__device__ __forceinline__ void after_previous()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Launches `kernel`, which calls after_previous(), to start early; in a stream
// that is being captured it is an ordinary launch (the graph then has only
// full dependencies, as its owner may expect) unless the library itself is
// capturing it (own_graph).  blocks > 0: prefer the shared-memory carve-out of so
// many blocks an SM, which leaves the rest to L1.
inline cudaError_t launch_early(const void *kernel, int grid, int block, void **args, size_t smem, cudaStream_t s,
                                bool own_graph = false, int blocks = 0)
{
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (!own_graph && cudaStreamIsCapturing(s, &capture) != cudaSuccess) {
        cudaGetLastError();  // the legacy stream while another one is being captured: the launch will say so
        capture = cudaStreamCaptureStatusNone;
    }
    cudaLaunchAttribute attrs[2] = {};
    int n = 0;
    if (capture == cudaStreamCaptureStatusNone) {
        attrs[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attrs[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (blocks > 0) {  // (1 KB a block is the system's; of the SM's 228 KB)
        const size_t percent = ((size_t)blocks * (smem + 1024) * 100 + 228 * 1024 - 1) / (228 * 1024);
        attrs[n].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
        attrs[n++].val.sharedMemCarveout = (unsigned)(percent < 100 ? percent : 100);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attrs;
    cfg.numAttrs = n;
    return cudaLaunchKernelExC(&cfg, kernel, args);
}

// List entries of BITS bits in a lane's words (32 words apart), as byte
// offsets of staged entries of 2^SHIFT bytes.
template <int BITS, int SHIFT = 4>
struct List {
    static constexpr uint32_t kPer = 32 / BITS;
    static __device__ __forceinline__ uint32_t in_word(uint32_t word, uint32_t j)
    {
        return ((word >> (BITS * j)) & ((1u << BITS) - 1u)) << SHIFT;
    }
    static __device__ __forceinline__ uint32_t at(const uint32_t *list, uint32_t t)
    {
        return in_word(list[32u * (t / kPer)], t % kPer);
    }
};

// Packed FP32 pairs: one instruction for two operations, the same roundings.
__device__ __forceinline__ uint64_t pair(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void halves(uint64_t v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// The larger of two, NaN when either is.
__device__ __forceinline__ float max_nan(float a, float b)
{
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// Words of the halo ids of a window, whole 16-byte copies.
__host__ __device__ inline uint32_t ids_words_of(const WindowShape &s) { return ((uint32_t)s.halo + 3u) & ~3u; }

}  // namespace sls
