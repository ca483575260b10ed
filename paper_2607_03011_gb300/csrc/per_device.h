// per_device.h -- values found out once per GPU (function attributes set, clusters that fit).
#pragma once
#include <mutex>

namespace isoloco {

// Function attributes and occupancy belong to a device: a process may hold plans on several, and
// make its first calls from several threads.
class PerDevice {
public:
    // *value for `device`, from make(value), which returns 0 or an error, the first time; an error
    // is returned and make runs again on the next call.  Devices past kMax are not remembered.
    template <class E, class F>
    E get(int device, int* value, F make) {
        if (device < 0 || device >= kMax) return make(value);
        std::lock_guard<std::mutex> lock(mutex_);
        if (!known_[device]) {
            const E e = make(&value_[device]);
            if (e != static_cast<E>(0)) return e;
            known_[device] = true;
        }
        *value = value_[device];
        return static_cast<E>(0);
    }

private:
    static constexpr int kMax = 64;
    std::mutex mutex_;
    bool known_[kMax] = {};
    int value_[kMax] = {};
};

}  // namespace isoloco
