// A yes-or-no property of the devices of a process, found once for each.
#pragma once

#include <atomic>

struct dsr_per_device {
    enum { DEVICES = 64 };  // devices beyond are asked each time
    std::atomic<signed char> known[DEVICES] = {};  // 0: not asked yet, 1: no, 2: yes

    // ask() finds the property of `device`. Threads that meet here on a
    // device's first use may each ask; they get the same answer.
    template <class Ask>
    bool get(int device, Ask ask) {
        if (device < 0 || device >= DEVICES) return ask();
        signed char k = known[device].load(std::memory_order_acquire);
        if (!k) {
            k = ask() ? 2 : 1;
            known[device].store(k, std::memory_order_release);
        }
        return k == 2;
    }
};
