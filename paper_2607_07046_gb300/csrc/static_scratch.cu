// Scratch of the ATTN decode step that allocates nothing: a fixed array of the module.
//
// The ordinary ATTN decode step keeps its intermediates (rotated queries, attention output) in
// per-device buffers that vt_partition_create allocated.  Callers that must not allocate device
// memory run the same kernels with those two vectors in one file-scope __device__ array, which the
// CUDA loader places in device memory together with the module's code, before any call.  The
// attention kernel (k_attn_decode) merges its slices in distributed shared memory, so the array
// holds nothing else and nothing in it has to start at zero: both vectors are written before they
// are read within a call.  (A split-K kernel of its own with its slice states in this array, 16
// slices of 4 warps per KV head, took 47.9 us at 2 KV heads and 4096 positions against 7.6 us.)
// Races: two calls in flight at once (two streams, or two host threads) share the one array and
// corrupt each other's intermediates; calls must be ordered.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "internal.h"

namespace vt {

static __device__ __align__(256) uint8_t g_static_scratch[kStaticScratchBytes];

static size_t round256(size_t b) { return (b + 255) & ~(size_t)255; }

StaticAttnLayout static_attn_layout(int hq, int hk, int dh) {
    StaticAttnLayout L{};
    L.q = 0;
    L.attn = round256((size_t)hq * dh * 4);
    // the call's published limit: 256 bytes and 16 slice states (max, sum, weighted V) per KV head more
    // than the two vectors take
    const size_t end = 256 + 2 * L.attn;
    const size_t group = (size_t)(hk > 0 ? hq / hk : 1), states = (size_t)hk * kStaticSplits * group;
    L.bytes = end + round256(states * 2 * 4) + round256(states * (size_t)dh * 4);
    return L;
}

// The device address of the array, looked up once per device (with that device current) and kept.
cudaError_t static_scratch_base(void** out) {
    static std::mutex mu;
    static void* addr[kStaticMaxDevices] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kStaticMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess) return e;
        if (!p) return cudaErrorInvalidSymbol;
        addr[dev] = p;
    }
    *out = addr[dev];
    return cudaSuccess;
}

}  // namespace vt
