// Bulk copies (cp.async.bulk, the TMA engine's 1-D form) and mbarrier waits
// for the staged kernels of the operator.  Every wait is bounded by the
// %globaltimer: a wait that gives up records SDP_ERR_TIMEOUT in the caller's
// status word and returns false, so a kernel never spins without end.
#pragma once

#include <cuda.h>
#include <stdint.h>

#include <atomic>

#include "sdp_internal.cuh"

namespace sdp {

// The current device and its number of SMs.
inline cudaError_t current_device(int& dev, int& nsm) {
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm < 1) {
        cudaGetLastError();
        return cudaErrorInvalidDevice;
    }
    return cudaSuccess;
}

// The dynamic shared-memory limit of one kernel instantiation, set on a device with the first
// launch there to the most that any launch takes.  The limit belongs to the kernel and the device:
// set to each launch's own bytes, another thread's smaller launch could lower it between this
// thread's setting and its launch, which is then refused.
class SharedLimit {
public:
    template <class K>
    cudaError_t raise(K kernel, int most, int dev) {
        if (dev < kDevices && set_[dev].load(std::memory_order_acquire)) return cudaSuccess;
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e != cudaSuccess)
            cudaGetLastError();
        else if (dev < kDevices)
            set_[dev].store(true, std::memory_order_release);
        return e;
    }

private:
    static constexpr int kDevices = 64;
    std::atomic<bool> set_[kDevices] = {};
};

// CTAs of one kernel instantiation with a fixed amount of shared memory that are resident at once
// on the current device, found once per device.
class ResidentCtas {
public:
    template <class K>
    cudaError_t get(K kernel, int bytes, int threads, long long& ctas) {
        int dev = 0, nsm = 0;
        cudaError_t e = current_device(dev, nsm);
        if (e != cudaSuccess) return e;
        int per_sm = dev < kDevices ? per_sm_[dev].load(std::memory_order_relaxed) : 0;
        if (per_sm == 0) {
            e = limit_.raise(kernel, bytes, dev);
            if (e != cudaSuccess) return e;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, bytes);
            if (e != cudaSuccess) return e;
            if (per_sm < 1) per_sm = 1;
            if (dev < kDevices) per_sm_[dev].store(per_sm, std::memory_order_relaxed);
        }
        ctas = (long long)nsm * per_sm;
        return cudaSuccess;
    }

private:
    static constexpr int kDevices = 64;
    SharedLimit limit_;
    std::atomic<int> per_sm_[kDevices] = {};
};

namespace tma {

constexpr unsigned long long kWaitNs = 1000000000ull;   // one second per wait

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Arrive (one of the barrier's expected arrivals) and add `bytes` to the
// transaction count the phase waits for.
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// Global -> shared copy of `bytes` (a multiple of 16; both addresses 16-byte
// aligned), completing as transaction bytes on `bar`.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// Store of a dense shared-memory box at coordinates (x, y, z, w) of a 4-D tensor map, parts
// outside the tensor left out, as one bulk group of the calling thread.  The box's writers
// have run fence_async, then a barrier with this thread.  x times the element size is a
// multiple of 16 bytes, no coordinate is negative.
__device__ __forceinline__ void tensor_store_4d(const CUtensorMap* map, const void* box, int x, int y, int z, int w) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"(map),
                 "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(box))
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// Load of the box at coordinates (x, y, z, w) of a 4-D tensor map into dense shared memory
// (128-byte aligned), completing as transaction bytes on `bar`.  x times the element size is a
// multiple of 16 bytes.
__device__ __forceinline__ void tensor_load_4d(const CUtensorMap* map, void* box, int x, int y, int z, int w,
                                               uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(smem_u32(box)),
        "l"(map), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar))
        : "memory");
}

// The same for a 3-D tensor map.
__device__ __forceinline__ void tensor_load_3d(const CUtensorMap* map, void* box, int x, int y, int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(smem_u32(box)),
        "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// The calling thread's writes to shared memory, before bulk operations that read them.
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// The calling thread's bulk groups have read their shared memory, which may be rewritten.
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// Wait for the phase of `bar` with parity `parity`; false after limit_ns (and
// the status word then holds SDP_ERR_TIMEOUT).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* status,
                                          unsigned long long limit_ns = kWaitNs) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = gtimer();
    while (!mbar_try_wait(bar, parity)) {
        if (gtimer() - t0 > limit_ns) {
            if (status) atomicCAS(status, 0, SDP_ERR_TIMEOUT);
            return false;
        }
    }
    return true;
}

}  // namespace tma
}  // namespace sdp
