// Host check of csrc/slots.h with a page of ordinary memory; prints one line
// per expectation that fails.
#include <cstdio>
#include <set>
#include <vector>

#include "slots.h"

static std::vector<double*> pages;
static bool mapped = true, none = false;
struct Fake {
    static double* alloc()
    {
        if (none) return nullptr;
        pages.push_back(new double[256]);
        mapped = true;
        return pages.back();
    }
    static bool alive(const double* p) { return mapped && p == pages.back(); }
};
static int bad = 0;
static void expect(bool ok, const char* what)
{
    if (!ok) {
        printf("%s\n", what);
        bad = 1;
    }
}

int main()
{
    cslbm::SlotPool<Fake> pool;
    none = true;
    expect(!pool.take().p, "no memory, no slot");
    none = false;
    std::vector<cslbm::Slot> got;
    std::set<double*> seen;
    for (int i = 0; i < 64; i++) {
        got.push_back(pool.take());
        expect(got[i].p >= pages[0] && got[i].p + 4 <= pages[0] + 256, "a slot lies in the page");
        seen.insert(got[i].p);
    }
    expect(seen.size() == 64 && pages.size() == 1, "64 slots of one page");
    cslbm::Slot over = pool.take();
    expect(!over.p, "the 65th context has none");
    pool.give(over);
    pool.give(got[17]);
    expect(pool.take().p == got[17].p, "a slot given back is taken again");
    for (auto& s : got) pool.give(s);
    expect(pool.take().p == got[0].p && pages.size() == 1, "the page is kept");
    // a device reset: the next take gets a new page, late gives of the old one change nothing
    mapped = false;
    cslbm::Slot a = pool.take();
    expect(pages.size() == 2 && a.p == pages[1], "a page no longer mapped is replaced");
    pool.give(got[0]);
    expect(pool.take().p == pages[1] + 4, "a slot of the old page is not given to the new one");
    return bad;
}
