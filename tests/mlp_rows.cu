// Host-only: the row offsets of the MLP's batch arrays do not wrap for any
// batch that an int32 counts.
#include <cstdio>

#include "../paper_2303_10581_gb300/csrc/mlp.cuh"

int main()
{
    using namespace ch::mlp;
    const long long B = 2147483647;
    const bool ok = row(B - 1, kIn) == (B - 1) * 1024 && row(33000000, kOut) == 2244000000ll &&
                    row(B - 1, kOut) == (B - 1) * 68 && row(B - 1, kHid) == (B - 1) * 64;
    std::printf(ok ? "rows ok\n" : "a row offset wraps\n");
    return ok ? 0 : 1;
}
