// tvl1_device_once.h -- what a process prepares once per device.  A kernel's attributes (its dynamic shared memory
// above 48 KB, non-portable cluster sizes) belong to one device, while contexts may live on any.
#pragma once
#include <mutex>

namespace tvl1 {

class DeviceOnce {
  public:
    // Runs prepare() at the first call with this device number; returns what it returned then.  Device numbers
    // beyond the table prepare at every call.
    template <typename F> int run(int device, F prepare) {
        if (device < 0 || device >= MAX_DEVICES) return prepare();
        std::call_once(once_[device], [&] { result_[device] = prepare(); });
        return result_[device];
    }

  private:
    static constexpr int MAX_DEVICES = 64;
    std::once_flag once_[MAX_DEVICES];
    int result_[MAX_DEVICES] = {};
};

}  // namespace tvl1
