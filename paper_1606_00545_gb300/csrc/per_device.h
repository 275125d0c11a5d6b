// per_device.h -- a set-up that every device needs once.  A kernel's function
// attributes belong to the device that was current when they were set, so "once
// per process" leaves a second device of the same process without them.  Host
// C++ only, without the CUDA headers.
#pragma once

#include <mutex>

namespace hec {

// get(device, f): the result of f() of the first call for that device, from any
// thread.
template <class R> class PerDevice {
public:
    template <class F> R get(int device, F &&f)
    {
        if (device < 0 || device >= kSlots)
            return f(); // (setting an attribute again is harmless)
        std::call_once(once_[device], [&]() { result_[device] = f(); });
        return result_[device];
    }

private:
    static constexpr int kSlots = 64;
    std::once_flag once_[kSlots];
    R result_[kSlots] = {};
};

} // namespace hec
