// Scratch of calls that have no handle, kept between calls: a call owns its slot
// from take() to keep(), so threads and streams never share one.  At most KEEP idle
// slots are kept on a device, and drain() hands them back to be freed.
#pragma once
#include <mutex>
#include <vector>

template <class Slot, int KEEP, int DEVICES>
class SlotPool {
    std::mutex mu;
    std::vector<Slot> idle[DEVICES];

public:
    // An idle slot of device dev; false: there is none, the caller makes one.
    bool take(int dev, Slot *s)
    {
        std::lock_guard<std::mutex> lk(mu);
        if (idle[dev].empty())
            return false;
        *s = idle[dev].back();
        idle[dev].pop_back();
        return true;
    }
    // Takes an unused slot back; false: enough are kept, the caller frees it.
    bool keep(int dev, const Slot &s)
    {
        std::lock_guard<std::mutex> lk(mu);
        if ((int)idle[dev].size() >= KEEP)
            return false;
        idle[dev].push_back(s);
        return true;
    }
    // All idle slots, for the caller to free.
    std::vector<Slot> drain()
    {
        std::lock_guard<std::mutex> lk(mu);
        std::vector<Slot> all;
        for (auto &v : idle) {
            all.insert(all.end(), v.begin(), v.end());
            v.clear();
        }
        return all;
    }
};
