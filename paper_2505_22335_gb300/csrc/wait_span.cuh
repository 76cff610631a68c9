// A caller's timeout in milliseconds as a duration that a clock can be advanced by.
// Plain C++, so that it can be run on the host too.
#pragma once

#include <chrono>

namespace ups {

// Infinity and everything above a year: a year.  wait_for converts to whole nanoseconds
// and adds them to now, which a larger number overflows (a deadline in the past).  Below
// zero and NaN: none.
inline std::chrono::nanoseconds wait_span(double ms) {
    constexpr double kYear = 365.0 * 86400e3;
    if (!(ms > 0.0)) return std::chrono::nanoseconds(0);
    return std::chrono::nanoseconds((long long)((ms < kYear ? ms : kYear) * 1e6));
}

}  // namespace ups
