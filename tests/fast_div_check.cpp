// Host build of the library's division by multiplication (csrc/fast_div.h) for
// the CPU test: for every divisor on the command line, compares with the
// division at multiples of it, next to them, and at the ends of the range.
#include <cstdio>
#include <cstdlib>

#include "fast_div.h"

int main(int argc, char** argv)
{
    const unsigned top = (1u << 28) - 1;
    for (int i = 1; i < argc; i++) {
        const unsigned d = (unsigned)strtoul(argv[i], nullptr, 10);
        const cslbm::Div q = cslbm::make_div(d);
        auto bad = [&](unsigned v) { return v <= top && cslbm::div_by(v, q) != v / d; };
        const unsigned step = d < 4096 ? d * (1 + 65536 / d) : d;
        for (unsigned long long m = 0; m <= top; m += step)
            for (int k = -2; k <= 2; k++)
                if ((long long)m + k >= 0 && bad((unsigned)(m + k))) return printf("%u / %u\n", (unsigned)(m + k), d), 1;
        for (unsigned v = 0; v < 70000; v++)
            if (bad(v) || bad(top - v)) return printf("%u or %u / %u\n", v, top - v, d), 1;
    }
    return 0;
}
