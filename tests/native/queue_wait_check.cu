// Host-only check of pic::queue_then_wait (field read-outs into the caller's memory) with a
// fake queue: every way in which one item, the wait or both can fail.  Exit status 0 when the
// wait has run once, after the last item, no item was queued behind a failure, and the first
// error is what the call returns.
#include <cstdio>

#include "../../paper_0909_5603_gb300/csrc/pic_internal.h"

int main()
{
    for (int n = 0; n <= 6; ++n)
        for (int bad = -1; bad < n; ++bad)
            for (int wait_fails = 0; wait_fails < 2; ++wait_fails) {
                int queued = 0, waits = 0, queued_at_wait = -1;
                const cudaError_t e = pic::queue_then_wait(
                    n,
                    [&](int i) {
                        if (i != queued) queued = 1000;  // out of order
                        ++queued;
                        return i == bad ? cudaErrorInvalidValue : cudaSuccess;
                    },
                    [&] {
                        ++waits;
                        queued_at_wait = queued;
                        return wait_fails ? cudaErrorUnknown : cudaSuccess;
                    });
                const int want_queued = bad < 0 ? n : bad + 1;
                const cudaError_t want = bad >= 0 ? cudaErrorInvalidValue : wait_fails ? cudaErrorUnknown : cudaSuccess;
                if (queued != want_queued || queued_at_wait != want_queued || waits != 1 || e != want) {
                    printf("n %d, item %d fails: %d queued, %d waits, error %d\n", n, bad, queued, waits, (int)e);
                    return 1;
                }
            }
    printf("queue_then_wait ok\n");
    return 0;
}
