// device_once.cuh -- what the host sets or asks once and keeps per device.
//
// A kernel's attributes and its occupancy hold for the device that is current when they are
// set or asked for. Kept under one flag for the whole process, a context on a second device
// launched kernels whose shared-memory limit had been raised on the first device only, which
// fails. Several host threads may come here at the same time; each then asks for itself.
#pragma once
#include <cuda_runtime_api.h>

#include <atomic>
#include <initializer_list>

namespace sparc {

class DeviceOnce {
public:
    // value = the positive number that ask(device, value) gave for the current device, asked for
    // again until it succeeds once (always, on devices beyond kDevices)
    template <typename F>
    cudaError_t get(int &value, F &&ask)
    {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const bool kept = dev >= 0 && dev < kDevices;
        value = kept ? known_[dev].load(std::memory_order_acquire) : 0;
        if (value > 0) return cudaSuccess;
        if ((e = ask(dev, value)) != cudaSuccess) return e;
        if (kept) known_[dev].store(value, std::memory_order_release);
        return cudaSuccess;
    }

    // `bytes` of dynamic shared memory for the kernels, on the current device
    template <typename... K>
    cudaError_t allow_smem(int bytes, K *...kernels)
    {
        int v;
        return get(v, [&](int, int &set) {
            cudaError_t e = cudaSuccess;
            for (const void *k : {(const void *)kernels...})
                if (e == cudaSuccess)
                    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
            set = 1;
            return e;
        });
    }

private:
    static constexpr int kDevices = 64;
    std::atomic<int> known_[kDevices] = {};
};

// n = the CTAs of `kernel`, of nt threads and no dynamic shared memory, that device `dev` holds at
// once (a cooperative launch's limit)
inline cudaError_t coop_blocks(const void *kernel, int nt, int dev, int &n)
{
    int sms = 0, per = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, nt, 0);
    n = sms * (per > 0 ? per : 1);
    return e;
}

}  // namespace sparc
