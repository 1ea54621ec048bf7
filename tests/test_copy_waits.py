"""Host run of the second stage's waits for its copies (CopyWait of
csrc/fe_waits.cuh, the code the kernel runs), a counter in the place of the
clock: a copy that never arrives ends the warp's copies and waits after one
limit (and one more before it leaves), however many items are left, and no copy
is asked for on a barrier whose phase is not over."""
from tests.test_fill_roles import run_host

PROGRAM = r"""
#include "fe_waits.cuh"
#include <cstdio>

int main() {
    const int items = 1000;
    const long limit = 50;
    int bad = 0;
    for (int lost : {0, 1, 7, 999, -1})                // the copy that never arrives (-1: all do)
        for (int other : {-1, 0, 5, 500}) {            // the item from which another warp's wait has given up
            fe::CopyWait cw;
            long tries = 0, t0 = 0;
            int asked = 0, got = 0, item = 0, overlapped = 0;
            unsigned phase = 0;                        // of the barrier: completed copies
            auto over_in = [&](long limit_from) { return tries - limit_from > limit; };
            auto ask = [&] {
                cw.ask([&] {
                    if (asked != (int)phase) overlapped++;
                    asked++;
                });
            };
            auto here = [&](unsigned parity) {
                tries++;
                // the copy on its way arrives at its third try, unless it is the lost one
                if (asked == (int)phase + 1 && asked - 1 != lost && tries % 3 == 0) phase++;
                return ((phase & 1u) ^ 1u) == parity;  // the phase of that parity is over
            };
            auto stop = [&] { return (other >= 0 && item >= other && asked - 1 == lost) || over_in(t0); };
            ask();
            for (item = 0; item < items; item++) {
                t0 = tries;
                if (cw.arrived(here, stop)) got++;
                if (item + 1 < items) ask();
            }
            const long before = tries;
            t0 = tries;
            cw.leave(here, [&] { return over_in(t0); });
            const int want = lost < 0 ? items : lost;
            const long most = 3L * want + 2 * (limit + 2) + 3;
            if (got != want || overlapped || asked != (lost < 0 ? items : lost + 1) || tries > most ||
                (lost < 0 && tries != before)) {
                bad++;
                std::printf("lost %d other %d: got %d asked %d overlapped %d tries %ld (most %ld)\n", lost, other, got, asked,
                            overlapped, tries, most);
            }
        }
    return bad ? 1 : 0;
}
"""


def test_a_lost_copy_costs_two_limits_at_most(tmp_path):
    run_host(tmp_path, PROGRAM)
