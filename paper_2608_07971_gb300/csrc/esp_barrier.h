// The word of the grid barrier of the grid-resident placement solve (internal; host and device, so that its
// arithmetic is tested on the CPU).
//
// One 64-bit word: bits 0 .. 62 count arrivals, bit 63 says that a CTA gave up waiting. Arrivals, the give-up
// and the polls are all 64-bit accesses of this one word: the memory model orders an acquire load after a
// release only where both are accesses of the same size at the same address, so two 32-bit words polled by
// one 64-bit load would carry no order. One word also keeps a poll to one trip to L2.
#pragma once

#include "esp_common.h"

namespace esp {

constexpr unsigned long long kBarAbort = 1ull << 63;

// Every byte of a held barrier (a test hook): the count about 2^61.6 arrivals short of zero and of every target,
// the abort bit clear.
constexpr int kBarHeldByte = 0x40;

// The count of v has reached target (both modulo 2^63, so that a held word stays short).
ESP_HD bool bar_reached(unsigned long long v, unsigned long long target)
{
    return (long long)((v - target) << 1) >= 0;
}

ESP_HD bool bar_aborted(unsigned long long v)
{
    return (v & kBarAbort) != 0;
}

}  // namespace esp
