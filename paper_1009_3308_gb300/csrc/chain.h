// Two launches that belong together: the second uses up what an earlier kernel
// left for both (the FP64 digit sums: the column exponents of the ring output,
// raised by atomic maxima and cleared by the finish).  Where one of them is not
// launched, reset() clears it instead, or the next call would start from it.
#pragma once

namespace sph {

template <typename First, typename Second, typename Reset>
inline int chain_or_reset(First&& first, Second&& second, Reset&& reset) {
    int rc = first();
    if (!rc) rc = second();
    if (rc) reset();
    return rc;
}

}  // namespace sph
