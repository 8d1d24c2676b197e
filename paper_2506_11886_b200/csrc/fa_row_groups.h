// Groups of batch rows that take turns in the room for block moments of one call.  Host arithmetic only: how each launch follows the
// one in front is decided here and can be checked without a device.
#pragma once
#include <cstddef>

namespace fa {

struct RowGroup {
    int b0, nb;              // batch rows b0 .. b0 + nb
    bool second;             // its moments go to the second half of the room
    bool wait_first;         // the launch in front may still read where its moments go
    bool chained;            // behind a launch of this call: it may begin while that one runs
};

// Calls launch(group) (0: go on) for groups of the B rows of a call, as many at a time as the room allows that holds the moments of `fit` (at least
// one) rows: all at once, or half of the room's rows by turns, or each where the one before was.  (Two halves are enough because a launch begins
// only when the one two in front of it has ended: the projection between them waits for the moments in front, whose end waits for that one.)  live(b): row b has moments.  A group
// without such a row launches nothing: it neither stands in front of another launch nor takes a turn.
template <typename Live, typename Launch>
int for_row_groups(int B, size_t fit, Live live, Launch launch) {
    const int group = fit >= (size_t)B ? B : fit >= 2 ? (int)(fit / 2) : 1;
    int launched = 0;
    for (int b0 = 0; b0 < B; b0 += group) {
        const int nb = B - b0 < group ? B - b0 : group;
        bool any = false;
        for (int b = b0; b < b0 + nb; ++b) any = any || live(b);
        if (!any) continue;
        const int err = launch(RowGroup{b0, nb, fit >= 2 && (launched & 1) != 0, fit < 2 && launched > 0, launched > 0});
        if (err) return err;
        ++launched;
    }
    return 0;
}

}  // namespace fa
