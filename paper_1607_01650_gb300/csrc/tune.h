// Choice between kernel variants by timing (host code, no CUDA).
#pragma once

#include <algorithm>

namespace dect {

// Time of a variant: the median of three samples, in which one disturbed launch
// does not count.  best: the least median so far.  The third sample is left out where the
// first two are both above best, as the median then is too, and the smaller of
// them is returned: which variant wins is what three samples each would give.
// sample(t) takes one and returns false to give up (then us is not set).
template <typename Sample>
bool median_time(float best, Sample sample, float &us)
{
    float a, b, c;
    if (!sample(a) || !sample(b)) return false;
    if (std::min(a, b) > best) {
        us = std::min(a, b);
        return true;
    }
    if (!sample(c)) return false;
    us = std::max(std::min(a, b), std::min(std::max(a, b), c));
    return true;
}

}  // namespace dect
