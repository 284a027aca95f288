// Host-only check (no GPU needed) of what a workspace carries from one call
// to the next: the records that kernels leave zeroed for the next call, and
// that no call zeroes, lie at the same place whatever n and the number of
// sets, outside the range that calls zero.  The counters of the speculative
// sample are among them: at a place that depends on n they would be other
// calls' data, and the sample's last block might never be elected.
#include <cstddef>
#include <cstdio>

#include "../paper_2303_10581_gb300/csrc/common.cuh"

using namespace ch;

int main()
{
    static_assert(offsetof(ExtCtrl, sample_done) < sizeof(ExtCtrl) && offsetof(ExtCtrl, sample_kmax) < sizeof(ExtCtrl),
                  "the sample's counters are in the record at a fixed place");
    int fails = 0;
    const Layout A = make_layout(1);
    for (int64_t n : {(int64_t)2, (int64_t)4097, (int64_t)1 << 22, ((int64_t)1 << 22) + 4097, (int64_t)100000007})
        for (int64_t sets : {0, 1, 4096}) {
            const Layout L = make_layout(n, sets);
            if (L.extctrl != A.extctrl || L.kxctrl != A.kxctrl || L.persist != A.persist ||
                L.extctrl + sizeof(ExtCtrl) > L.ctrl || L.kxctrl + sizeof(KxCtrl) > L.ctrl) {
                std::printf("n=%lld sets=%lld: a self-resetting record moves\n", (long long)n, (long long)sets);
                ++fails;
            }
        }
    if (!fails) std::printf("reuse ok\n");
    return fails ? 1 : 0;
}
