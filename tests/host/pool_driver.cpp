// Host-only driver for efm::WorkPools (which pool a work area comes from), used
// by tests/test_pools.py: a fake of the CUDA calls, one command a line on
// stdin, one line of output a command.
//   ctx I       the current context (0: none)
//   fail 0|1    whether making a pool fails
//   get         -> pool P (0: the default pool)
#include <cstdio>
#include <cstring>

#include "efm_pool.h"

static unsigned long long g_ctx = 0;
static int g_fail = 0, g_made = 0;

struct FakeApi {
    using Pool = int *;
    bool context(uint64_t &id)
    {
        id = g_ctx;
        return g_ctx != 0;
    }
    Pool create() { return g_fail ? nullptr : new int(++g_made); }
};

int main()
{
    static efm::WorkPools<FakeApi> pools;
    char cmd[16];
    while (std::scanf("%15s", cmd) == 1) {
        if (!std::strcmp(cmd, "ctx")) {
            if (std::scanf("%llu", &g_ctx) != 1) return 2;
            std::printf("ok\n");
        } else if (!std::strcmp(cmd, "fail")) {
            if (std::scanf("%d", &g_fail) != 1) return 2;
            std::printf("ok\n");
        } else if (!std::strcmp(cmd, "get")) {
            int *p = pools.get();
            std::printf("pool %d\n", p ? *p : 0);
        } else {
            return 2;
        }
    }
    return 0;
}
