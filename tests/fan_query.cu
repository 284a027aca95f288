// Host-only: prints what tests of the hull step's fan need to know of the
// library's own constants and workspace: the bin counts of both levels, and
// (arguments: workspace bytes, sets) where ch_hull_batched counts each set's
// points to sort.
#include <cstdio>
#include <cstdlib>

#include "../paper_2303_10581_gb300/csrc/common.cuh"

using namespace ch;

int main(int argc, char **argv)
{
    unsigned long long soct = 0;
    if (argc > 2) {
        const size_t bytes = std::strtoull(argv[1], nullptr, 10);
        const int64_t sets = std::strtoll(argv[2], nullptr, 10);
        int64_t lo = 0, hi = kMaxHullN - 1;   // the most points the workspace holds, as the call finds it
        while (lo < hi) {
            const int64_t mid = lo + (hi - lo + 1) / 2;
            if (make_batch_layout(make_layout(mid, sets), sets).total <= bytes) lo = mid;
            else hi = mid - 1;
        }
        soct = make_batch_layout(make_layout(lo < 1 ? 1 : lo, sets), sets).soct;
    }
    std::printf("%d %d %llu\n", kFanBins, kFan2Bins, soct);
    return 0;
}
