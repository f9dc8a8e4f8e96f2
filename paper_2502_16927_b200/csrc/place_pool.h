// A few places of static device memory that handles take and give back, on every device.  Host code without a CUDA header: the
// device calls come in as `Api` (int get(int*), int set(int), int synchronize(); 0 = success), so that the rules run on the CPU too.
#pragma once
#include <mutex>

namespace bigmac {

// Makes `device` the current one for its lifetime.
template <typename Api>
struct OnDevice {
    int before = -1;
    bool ok;
    explicit OnDevice(int device) : ok(Api::get(&before) == 0) {
        if (ok && before != device) ok = Api::set(device) == 0;
        else before = -1;
    }
    ~OnDevice() { if (before >= 0) Api::set(before); }
    OnDevice(const OnDevice&) = delete;
    OnDevice& operator=(const OnDevice&) = delete;
};

template <int DEVICES, int PLACES>
class PlacePool {
    std::mutex mutex;
    bool taken[DEVICES][PLACES] = {};

public:
    // A free place of the device: its number, or -1.
    int take(int device) {
        if (device < 0 || device >= DEVICES) return -1;
        std::lock_guard<std::mutex> lock(mutex);
        for (int i = 0; i < PLACES; ++i)
            if (!taken[device][i]) { taken[device][i] = true; return i; }
        return -1;
    }
    // Nothing of the holder may run when another takes the place: the device whose memory it is finishes its work first.  Where it
    // does not say so (a capture in progress, an earlier fault) the place stays taken.
    template <typename Api>
    bool give(int device, int place) {
        OnDevice<Api> on(device);
        if (!on.ok || Api::synchronize() != 0) return false;
        std::lock_guard<std::mutex> lock(mutex);
        taken[device][place] = false;
        return true;
    }
    // A place that nothing has used yet.
    void give_unused(int device, int place) {
        std::lock_guard<std::mutex> lock(mutex);
        taken[device][place] = false;
    }
};

}  // namespace bigmac
