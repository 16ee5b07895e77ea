// What a process does once per device ordinal (a kernel's attributes, a device's properties): they apply to the device
// that is current when they are made or asked for.
#pragma once
#include <atomic>

namespace hydra {

constexpr int kMaxDevices = 64;

// f() is run for device `dev` until it has returned 0 (success) once. Any number of host threads may call at the same time:
// several may then run f, which has to be harmless.
class OncePerDevice {
public:
    template <class F>
    auto operator()(int dev, F f) -> decltype(f())
    {
        using Status = decltype(f());
        if (done_[dev].load(std::memory_order_acquire)) return Status{};
        const Status status = f();
        if (status == Status{}) done_[dev].store(true, std::memory_order_release);
        return status;
    }

private:
    std::atomic<bool> done_[kMaxDevices] = {};
};

}  // namespace hydra
