// per_device.h -- what a launcher works out once per device and process: the
// device's SMs and a kernel's resident CTAs on each.  Host code only.
#pragma once

#include <atomic>
#include <cstdint>

namespace sl {

struct Residency {
    int sms = 0;      // SMs of the device
    int per_sm = 0;   // resident CTAs of the kernel on one SM, at least 1
};

// One Residency per device.  Both numbers are published in one word, so that a
// thread that finds a device ready has both and what was set up before them;
// threads that meet on an unready device all work it out, to the same values.
class ResidencyCache {
public:
    static constexpr int kDevices = 64;

    bool get(int dev, Residency &r) const
    {
        const uint64_t w = word_[dev].load(std::memory_order_acquire);
        r.sms = (int)(w >> 32);
        r.per_sm = (int)(uint32_t)w;
        return w != 0;
    }
    void set(int dev, const Residency &r)
    {
        word_[dev].store((uint64_t)(uint32_t)r.sms << 32 | (uint32_t)r.per_sm, std::memory_order_release);
    }

private:
    std::atomic<uint64_t> word_[kDevices] = {};
};

}  // namespace sl
