// Host side of the convolution layer's launches that needs no CUDA: what is known of each device.
#pragma once
#include <mutex>

namespace wici {

// SMs of a device, and its resident clusters of 1, 2, 4 and 8 CTAs (0: none fits).
struct ConvDevice {
    int sms = 0, clusters[4] = {};
};

// Every device is asked once (those past the table on each call); a caller gets a copy of its own
// device's entry, so that calls on several devices from several threads do not see one another's.
class ConvDevices {
public:
    // query(&d) fills d and returns 0, or an error, which is returned (and the device asked again)
    template <class Query>
    auto get(int dev, ConvDevice *out, Query query) -> decltype(query(out)) {
        std::lock_guard<std::mutex> lk(mu_);
        const bool kept = dev >= 0 && dev < kDevices;
        if (!kept || !known_[dev]) {
            ConvDevice d;
            if (const auto e = query(&d)) return e;
            *out = d;
            if (!kept) return {};
            table_[dev] = d;
            known_[dev] = true;
        }
        *out = table_[dev];
        return {};
    }

private:
    static constexpr int kDevices = 64;
    std::mutex mu_;
    bool known_[kDevices] = {};
    ConvDevice table_[kDevices];
};

}  // namespace wici
