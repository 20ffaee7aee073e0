// Host-only check of pic::sub_range_from (the walk by which the particle kernel finds the
// source sub-range of a slot): against a linear search on consistent tables, and, on tables
// that do not hold the slot asked for, that no entry outside the table is read.  The entries
// around a table are traps: values that a walk reading them would follow.  Exit status 0 when
// all agree.
#include <cstdio>

#include "../../paper_0909_5603_gb300/csrc/pic_internal.h"

constexpr int kMax = 64, kPad = 256;

static unsigned long long state = 0x243F6A8885A308D3ULL;
static int below(int n)
{
    state = state * 6364136223846793005ULL + 1442695040888963407ULL;
    return (int)((state >> 33) % (unsigned long long)n);
}

int main()
{
    static int mem[kPad + kMax + 1 + kPad];
    int *slot = mem + kPad;
    for (int n = 1; n <= kMax; ++n)
        for (int t = 0; t < 200; ++t) {
            for (int i = -kPad; i <= kMax + kPad; ++i) slot[i] = -1;
            slot[0] = below(2) ? 0 : 1024 * below(40);  // (a part's table starts at its first slot)
            for (int i = 1; i < n; ++i) slot[i] = slot[i - 1] + 1 + below(40);
            slot[n] = pic::kSlotEnd;
            const int first = slot[0], end = slot[n - 1] + 1 + below(40);
            // every slot, from every start that the warp's vote can give
            for (int p = first; p < end; ++p) {
                int want = 0;
                while (want + 1 < n && slot[want + 1] <= p) ++want;
                int at = -1;
                const int got = pic::sub_range_from(slot, below(want + 1), p, at);
                if (got != want || at != slot[want]) {
                    printf("n %d slot %d: sub-range %d, not %d\n", n, p, got, want);
                    return 1;
                }
            }
            // slots that the table does not hold: a population above the records', and a slot
            // before the first (a vote without a hit)
            const int odd[] = {end, end + 1, end + 255, first - 1, 0, 0x7ffffff0};
            for (int p : odd) {
                int at = -1;
                const int e = pic::sub_range_from(slot, below(n + 1) - 1, p, at);
                if (e < 0 || e >= n || at != slot[e]) {
                    printf("n %d slot %d beyond %d: sub-range %d\n", n, p, end, e);
                    return 1;
                }
            }
        }
    printf("sub_range_from ok\n");
    return 0;
}
