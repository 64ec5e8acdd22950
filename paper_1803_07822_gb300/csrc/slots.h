// Slots of mapped host memory the reductions write their result to: 64 of four
// doubles in one page of the process, taken by a context's first reduction and
// given back by cslbm_destroy.  The page is kept for the contexts to come; one
// that a device reset has ended (its addresses are no longer mapped, and a
// kernel that wrote there would fault) is noticed by the next take and replaced.
#pragma once

#include <mutex>

namespace cslbm {

struct Slot {
    double* p = nullptr;    // four doubles, or null: none free, or no mapped memory
    unsigned long long page = 0;  // the page it is of, by count
};

// Memory: alloc() a page of 64 x 4 doubles or null; alive(page) whether it is still mapped
template <class Memory> class SlotPool {
public:
    Slot take()
    {
        std::lock_guard<std::mutex> lock(mu);
        if (page && !Memory::alive(page)) page = nullptr;
        if (!page) {
            page = Memory::alloc();
            used = 0;
            count++;
        }
        Slot s;
        for (int i = 0; page && i < 64; i++)
            if (!(used >> i & 1)) {
                used |= 1ull << i;
                s.p = page + 4 * i;
                s.page = count;
                break;
            }
        return s;
    }
    void give(const Slot& s)
    {
        std::lock_guard<std::mutex> lock(mu);
        if (s.p && s.page == count) used &= ~(1ull << ((s.p - page) / 4));
    }

private:
    std::mutex mu;
    double* page = nullptr;
    unsigned long long used = 0, count = 0;
};

}  // namespace cslbm
