// Division by a divisor that is used many times: five dependent operations and no special cases, against
// 580 cycles for `/` in a chain of dependent prices, where a zero dividend takes its slow path (internal).
#pragma once

#include <cmath>

#include "esp_common.h"

namespace esp {

// a / b correctly rounded to nearest, given y = 1 / b correctly rounded. P. Markstein, "Computation of
// elementary functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34 (1990): if q is a
// faithful rounding of a / b and r = a - b q (exact in one fused multiply-add), then q + r y rounds to
// a / b rounded. a y alone may be off by more than one unit in the last place, so one step makes it
// faithful and the second makes it correct. Holds while neither q nor r leaves the normal range; here b is
// a capacity in [1, 2^63) and a is zero or 2^-900 <= |a| <= 2^1000 (see div_safe), so both stay inside.
ESP_HD double div_by(double a, double b, double y)
{
    double q = a * y;
    double r = fma(-b, q, a);
    q = fma(r, y, q);
    r = fma(-b, q, a);
    return fma(r, y, q);
}

// Whether div_by may divide a (a >= 0, given by its bits): zero, or from 2^-900 to below 2^1000.
ESP_HD bool div_safe(long long bits)
{
    return bits == 0 || (bits >= (123LL << 52) && bits < (2023LL << 52));
}

}  // namespace esp
