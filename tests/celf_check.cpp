// Reads k, before[k], after, gains[k] per line; prints the first mismatch.
#include <stdio.h>

#include <vector>

#include "sg_celf_check.h"

int main()
{
    int k;
    while (scanf("%d", &k) == 1) {
        std::vector<long long> before((size_t)k);
        std::vector<int64_t> gains((size_t)k);
        long long after = 0, x;
        for (auto &v : before)
            if (scanf("%lld", &v) != 1) return 1;
        if (scanf("%lld", &after) != 1) return 1;
        for (auto &v : gains) {
            if (scanf("%lld", &x) != 1) return 1;
            v = x;
        }
        printf("%d\n", sgi::celf_first_mismatch(before.data(), after, gains.data(), k));
    }
    return 0;
}
