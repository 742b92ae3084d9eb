// kept.h -- pinned blocks of one size kept for the next taker, per device.
#pragma once

#include <stdint.h>

#include <mutex>

namespace wt {

// At most kKept blocks a device, each of the context it was allocated in: a
// device's blocks are dropped, not freed, once its context is another (the old
// one is gone, and its pinned memory with it). What keep() refuses its caller
// frees. Nothing is allocated here, so nothing throws.
class Kept {
public:
    static constexpr int kDevices = 64, kKept = 32;

    void* take(int device, uint64_t ctx)
    {
        if (device < 0 || device >= kDevices) return nullptr;
        std::lock_guard<std::mutex> lk(mu_);
        Slot& s = slot_[device];
        if (s.ctx != ctx || s.n == 0) return nullptr;
        return s.p[--s.n];
    }

    bool keep(int device, uint64_t ctx, void* p)
    {
        if (device < 0 || device >= kDevices || ctx == 0) return false;
        std::lock_guard<std::mutex> lk(mu_);
        Slot& s = slot_[device];
        if (s.ctx != ctx) {
            s.ctx = ctx;
            s.n = 0;
        }
        if (s.n == kKept) return false;
        s.p[s.n++] = p;
        return true;
    }

private:
    struct Slot {
        uint64_t ctx = 0;
        int n = 0;
        void* p[kKept];
    };
    std::mutex mu_;
    Slot slot_[kDevices];
};

}  // namespace wt
