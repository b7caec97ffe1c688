// cluster.h -- size of a thread-block cluster (host only, no CUDA).
#pragma once

namespace mg {

// The largest cluster of want, want / 2, .. CTAs that resident(ctas) finds room
// for.  One CTA needs no cluster and always runs.
template <class Resident>
int cluster_step_down(int want, Resident resident)
{
    int c = want;
    while (c > 1 && !resident(c)) c /= 2;
    return c > 1 ? c : 1;
}

}  // namespace mg
