// Host build of AUTO's choice (rows::best_pass): reads lines "n0 n1 n2 yper
// zper s_bytes" and prints for each flat, rows or fused.
#include <cstdio>

#include "rows_plan.h"

int main()
{
    int n[3], yper, zper, sb;
    while (scanf("%d %d %d %d %d %d", n, n + 1, n + 2, &yper, &zper, &sb) == 6) {
        cslbm::rows::Plan pl{};
        const char* name[3] = {"flat", "rows", "fused"};
        const bool ok = cslbm::rows::make_plan(n, yper != 0, zper != 0, sb, 232448, pl);
        puts(ok ? name[cslbm::rows::best_pass(pl, n, sb, zper != 0)] : "flat");
    }
    return 0;
}
