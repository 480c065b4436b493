// host_wait.cuh -- the library's bounded host wait on the GPU.
#pragma once
#include <chrono>
#include <thread>

#include "common.cuh"

namespace ooc {

// Waits for `ev` by polling it: OOC_E_TIMEOUT once `timeout_ms` have passed
// (what was enqueued still runs).  The first two milliseconds are polled
// without sleeping, since a sleep of 20 us takes about 75 with the timer's
// slack: a call of a few hundred microseconds (ooc_compress_var waits once)
// would spend a tenth of its time asleep after the GPU is done.
inline ooc_status wait_event(cudaEvent_t ev, int64_t timeout_ms)
{
    const auto start = std::chrono::steady_clock::now();
    for (;;) {
        const cudaError_t e = cudaEventQuery(ev);
        if (e == cudaSuccess)
            return OOC_OK;
        if (e != cudaErrorNotReady)
            return OOC_E_CUDA;
        const auto t = std::chrono::steady_clock::now() - start;
        if (t > std::chrono::milliseconds(timeout_ms))
            return OOC_E_TIMEOUT;
        if (t > std::chrono::milliseconds(2))
            std::this_thread::sleep_for(std::chrono::microseconds(20));
    }
}

}  // namespace ooc
