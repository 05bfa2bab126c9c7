// deferred.h -- the order of a call whose steps leave the sums of their forces to later launches (host only).
#pragma once

namespace lbm {

// Runs `n` steps and sums the forces of up to `most` of them at once.  step(k, held) launches step k, whose
// partials go to place `held` of the unsummed ones; sum(held) sums those.  Both return 0 or an error code.  A
// step that fails ends the call, but the steps before it have run: their forces are summed all the same.  *lost is
// set to the number of steps that ran and whose forces could not be summed.
template <class Step, class Sum>
int run_deferred(long n, int most, Step&& step, Sum&& sum, int* lost) {
    int held = 0;
    *lost = 0;
    for (long k = 0; k < n; ++k) {
        int rc = step(k, held);
        const bool ran = rc == 0;
        if (ran) ++held;
        if (held > 0 && (!ran || held == most || k + 1 == n)) {
            const int rs = sum(held);
            if (rs) *lost = held;
            if (!rc) rc = rs;
            held = 0;
        }
        if (rc) return rc;
    }
    return 0;
}

}  // namespace lbm
