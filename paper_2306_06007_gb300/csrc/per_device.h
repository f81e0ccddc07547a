// Set-up that CUDA keeps per device (kernel attributes), done once on each: a process may hold plans on
// several GPUs.
#pragma once

#include <atomic>
#include <cstdint>

namespace hvox {

class OncePerDevice {
    static constexpr int kDevices = 256;
    std::atomic<uint64_t> done_[kDevices / 64] = {};

public:
    // Runs f unless it has returned for this device before. f can run twice (threads that meet here, a
    // device beyond the table), so it only sets what it would set again.
    template <class F> void run(int device, F f) {
        const bool known = device >= 0 && device < kDevices;
        const uint64_t bit = uint64_t(1) << (device & 63);
        if (known && (done_[device / 64].load() & bit)) return;
        f();
        if (known) done_[device / 64].fetch_or(bit);
    }
};

}  // namespace hvox
