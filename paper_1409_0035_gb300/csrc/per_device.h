// A value per CUDA device, made at its first use there (host code only).
// Kernel attributes and residency belong to a device, and a program may use
// several, from several threads.
#pragma once
#include <mutex>

namespace ccg {

template <class T> class PerDevice {
public:
    static constexpr int kMax = 64;
    // The value of device `dev`: make(T &) fills it and returns a status, whose
    // zero keeps it.  Devices beyond kMax make it every time.
    template <class Make> int get(int dev, T *out, Make make)
    {
        if (dev < 0 || dev >= kMax) return make(*out);
        std::lock_guard<std::mutex> lock(mu_);
        if (!have_[dev]) {
            T v{};
            const int rc = make(v);
            if (rc != 0) return rc;
            of_[dev] = v;
            have_[dev] = true;
        }
        *out = of_[dev];
        return 0;
    }

private:
    std::mutex mu_;
    T of_[kMax] = {};
    bool have_[kMax] = {};
};

// CTAs of a kernel that a device holds at once.
struct Residency {
    int per_sm = 0, sms = 0;
};

}  // namespace ccg
