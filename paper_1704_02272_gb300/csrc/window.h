// Window filter of a pattern set (see table.h): chosen and built on the host.
#pragma once
#include <stdint.h>

#include <vector>

namespace pfac {

struct WinPat {
    const uint8_t *p;
    uint32_t len;
};

struct WindowFilter {
    uint32_t words = 0, rep = 0, stride = 0, nb = 0, gw = 0, glen = 0, packed = 0, shorts = 0;
    std::vector<uint32_t> H;
};

// Picks the filter with the least estimated cost for uniform text and builds
// it; false when none is estimated to pay.  dens_f: share of uniform windows
// that pass the prefix bitmap the scan tests candidates against.
bool build_window_filter(const std::vector<WinPat> &pats, uint32_t sigma, uint32_t bps, double dens_f,
                         WindowFilter *out);

}  // namespace pfac
