// How many Monte Carlo dropout passes of one batch run side by side.
#pragma once

#include <algorithm>

#include "../../include/hyb.h"

namespace hyb {

// As many of `passes` as keep a launch's volume within max_cells (a small batch
// does not fill the SMs: 65 536 cells, four passes side by side, 6.3 -> 1.9 ms
// for 16), or fewer where reserve(n), which takes the buffers of n passes,
// answers HYB_ENOMEM: a batch whose single pass fits always runs.  cells >= 1.
template <class Reserve>
int passes_side_by_side(int passes, long long cells, long long max_cells, Reserve reserve) {
    int n = (int)std::max<long long>(1, std::min<long long>(passes, max_cells / cells));
    while (reserve(n) == HYB_ENOMEM && n > 1) n = (n + 1) / 2;
    return n;
}

}  // namespace hyb
