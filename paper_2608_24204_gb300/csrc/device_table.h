// What the library knows of each device (no CUDA needed).
#pragma once
#include <mutex>

namespace wici {

// Every device is asked once (those past the table on each call); a caller gets a copy of its own
// device's entry, so that calls on several devices from several threads do not see one another's.
template <class Counts>
class DeviceTable {
public:
    // query(&d) fills d and returns 0, or an error, which is returned (and the device asked again)
    template <class Query>
    auto get(int dev, Counts *out, Query query) -> decltype(query(out)) {
        std::lock_guard<std::mutex> lk(mu_);
        const bool kept = dev >= 0 && dev < kDevices;
        if (!kept || !known_[dev]) {
            Counts d;
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
    Counts table_[kDevices];
};

}  // namespace wici
