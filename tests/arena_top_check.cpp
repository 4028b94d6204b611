// Drives FreeList::alloc_top (arena.h): commands as in arena_check.cpp, and
//   top B     -> the offset, or -1 when nothing fits
#include <cstdio>
#include <cstring>

#include "arena.h"

int main()
{
    ising::FreeList f;
    char cmd[16];
    long long a = 0, b = 0;
    while (std::scanf("%15s", cmd) == 1) {
        if (!std::strcmp(cmd, "reset") && std::scanf("%lld", &a) == 1) {
            f.reset(a);
        } else if (!std::strcmp(cmd, "alloc") && std::scanf("%lld", &a) == 1) {
            std::printf("%lld\n", (long long)f.alloc(a));
        } else if (!std::strcmp(cmd, "top") && std::scanf("%lld", &a) == 1) {
            std::printf("%lld\n", (long long)f.alloc_top(a));
        } else if (!std::strcmp(cmd, "free") && std::scanf("%lld %lld", &a, &b) == 2) {
            f.release(a, b);
        } else {
            return 1;
        }
    }
    std::printf("%lld %zu\n", (long long)f.used, f.free_.size());
    return 0;
}
