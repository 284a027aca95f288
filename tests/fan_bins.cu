// Host-only: which bins have neighbours on both sides, also for the bin before
// the first that a point straight below the centre may be given.
#include <cstdio>

#include "../paper_2303_10581_gb300/csrc/fan.cuh"

int main()
{
    for (uint32_t nb : {512u, 1024u, 8192u, 27648u}) {
        const uint32_t in[] = {1u, 2u, nb / 2, nb - 3, nb - 2}, out[] = {0xffffffffu, 0xfffffffeu, 0u, nb - 1, nb, nb + 1};
        for (uint32_t b : in)
            if (!ch::inner_bin(b, nb)) return std::printf("bin %u of %u has neighbours\n", b, nb), 1;
        for (uint32_t b : out)
            if (ch::inner_bin(b, nb)) return std::printf("bin %d of %u has not\n", (int)b, nb), 1;
    }
    std::printf("bins ok\n");
    return 0;
}
