// tickets_ahead of perm_parts.h: prints its value for each "left walks most" of the input.
#include <cstdio>

#include "perm_parts.h"

int main() {
    long long left, walks;
    unsigned most;
    while (std::scanf("%lld %lld %u", &left, &walks, &most) == 3)
        std::printf("%u\n", perm::tickets_ahead(left, walks, most));
    return 0;
}
