// Choice and construction of the window filter (table.h, kernels_w.cuh).
//
// The free parameters are the stride S (how many starts one lookup covers),
// the symbols hashed, the bits tested per word, and how the shared memory is
// split between more words (fewer false candidates) and more copies (fewer
// bank conflicts).  Each combination is costed from the pattern lengths alone
// and only the best is built.
#include "window.h"

#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "internal.h"
#include "table.h"

namespace pfac {

namespace {

// Most strings inserted (completions of short patterns included).
constexpr double MAX_STRINGS = 2.0e6;
// Estimated SM cycles per slice above which the other scan kernels are used:
// one line for alphabets of 17 symbols on, one below.  64 MiB of uniform text,
// patterns of 4 to 64 symbols, this kernel / the faster of the others (the
// estimate): 20 symbols x 100,000 398 / 2,607 us (356); 256 x 100,000 93 / 331
// (150); 64 x 300,000 324 / 2,556 (781); 64 x 500,000 646 / 3,004 (1,850);
// 256 x 500,000 595 / 1,029 (1,816); 256 x 1,000,000 1,231 / 2,049 (3,680); 20
// x 300,000 from 6 symbols on 922 / 3,787 (726).  Packets, 50,000 signatures:
// 232 / 532 (422).  Small alphabets, whose few hashed symbols say less while
// the other kernels' filters see more of them: 4 x 300,000 from 14 symbols on
// 215 / 1,086 (494), but 10 x 20,000 from 5 on 733 / 599 (640) and 8 x 30,000
// from 6 on 1,304 / 234 (2,398).
constexpr double MAX_COST = 4000.0;
constexpr double MAX_COST_SMALL = 600.0;  // up to 16 symbols

struct Shape {
    uint32_t S, gw, g5, nb;
};

}  // namespace

bool build_window_filter(const std::vector<WinPat> &pats, uint32_t sigma, uint32_t bps, double dens_f,
                         WindowFilter *out) {
    if (pats.empty() || bps < 2) return false;
    const bool packed = bps == 2;
    const double A = (double)(1u << bps);
    uint32_t min_len = 0xFFFFFFFFu;
    std::vector<uint32_t> by_len(64, 0);  // patterns by length (63: that or more)
    for (const WinPat &p : pats) {
        min_len = std::min(min_len, p.len);
        by_len[std::min<uint32_t>(p.len, 63)]++;
    }
    // matches per start of a uniform text: every one is a candidate
    double match = 0;
    for (uint32_t L = 1; L < 64; L++) match += by_len[L] * pow((double)sigma, -(double)L);
    match = std::min(match, 1.0);

    std::vector<Shape> shapes;
    for (uint32_t S : {1u, 2u, 4u, 8u, 16u}) {
        if (S > min_len) break;
        if (packed) {
            for (uint32_t gw = 8; gw <= 14; gw++)
                for (uint32_t nb = 1; nb <= 2; nb++) shapes.push_back({S, gw, 0, nb});
        } else {
            for (uint32_t nb = 1; nb <= 3; nb++) {
                if (nb == 1) shapes.push_back({S, 2, 0, nb});
                for (uint32_t gw = 3; gw <= 4; gw++) shapes.push_back({S, gw, 0, nb});
                if (S == 1 && nb == 2) shapes.push_back({S, 5, 1, nb});
            }
        }
    }
    // powers of the symbol counts
    std::vector<double> a_pow(64, 1.0), s_pow(64, 1.0);
    for (int i = 1; i < 64; i++) {
        a_pow[i] = a_pow[i - 1] * A;
        s_pow[i] = s_pow[i - 1] / (double)sigma;
    }
    double best = bps > 4 ? MAX_COST : MAX_COST_SMALL;
    bool found = false;
    for (const Shape &s : shapes) {
        uint32_t glen = s.gw;
        for (uint32_t b = 0; b < s.nb; b++)
            glen = std::max(glen, win_off(packed, b) + (packed ? 3u : 1u));
        // strings inserted, and of them those whose word fills up (the free
        // symbols include the tested bits)
        double ins = 0, full = 0, real = 0;
        for (uint32_t L = 1; L < 64; L++) {
            if (!by_len[L]) continue;
            for (uint32_t o = 0; o < s.S; o++) {
                const uint32_t known = L > o ? std::min(L - o, glen) : 0u;
                const double n = by_len[L] * a_pow[glen - known];
                ins += n;
                real += by_len[L] * s_pow[known];
                if (!packed && known < glen && known >= s.gw) full += by_len[L];
            }
        }
        if (ins > MAX_STRINGS) continue;
        real = std::min(real, 1.0);
        for (uint32_t words : {49152u, 32768u, 16384u, 8192u, 4096u, 2048u, 1024u}) {
            const uint32_t reps = words > 32768 ? 0u : 0xFFFFFFFFu;
            uint32_t rep = 0;
            while (reps && (words << (rep + 1)) <= 32768u && rep < 5) rep++;
            // windows that pass without being in the set: Poisson strings per
            // word, each setting nb random bits; words that fill up count as
            // 32 single bits
            const double part = full > 0 ? full * 32.0 : 0.0;
            const double mu = (full > 0 ? (ins - full * A) : ins) / words;
            double fp = 0;
            if (s.nb == 1) {
                fp = 1.0 - exp(-(mu * words + part) / (32.0 * words));
            } else {
                if (mu > 30.0) {
                    fp = pow(1.0 - pow(31.0 / 32.0, mu * s.nb), (double)s.nb);
                } else {
                    double pn = exp(-mu), clear = 1.0;  // clear: a bit none of n strings set
                    const double keep = s.nb == 2 ? 961.0 / 1024.0 : 29791.0 / 32768.0;  // (31/32)^nb
                    for (int n = 0; n < 200; n++) {
                        const double set = 1.0 - clear;
                        fp += pn * (s.nb == 2 ? set * set : set * set * set);
                        pn *= mu / (n + 1);
                        clear *= keep;
                        if (n > mu && pn < 1e-9) break;
                    }
                }
                if (full > 0) fp += 1.0 - exp(-full / words);
            }
            const double pass = std::min(1.0, real + fp);
            const double L = 16.0 / s.S;
            const double alu = 16.0 + (packed ? 4.0 : 0.0) +
                               L * (8.0 + 2.0 * (s.nb - 1) + s.g5) / 4.0 * 1.2;
            const double lds = L * LOAD_WAVEFRONTS[rep] * 1.05;
            const double cand = 512.0 / s.S * pass;
            // starts left after the prefix bitmap
            const double left = 512.0 * match +
                                std::min(cand * s.S * dens_f, 512.0 * dens_f);
            // filling shared memory at 64 bytes a cycle, spread over a
            // thousand slices per SM
            const double fill = (double)(words << rep) * 4.0 / 64.0 / 1000.0;
            const double cost = std::max(alu, lds) + cand * (2.0 + 3.0 * s.S) + left * 10.0 + fill;
            if (cost < best) {
                best = cost;
                found = true;
                out->words = words;
                out->rep = rep;
                out->stride = s.S;
                out->nb = s.nb;
                out->gw = s.gw;
                out->glen = glen;
                out->packed = packed;
                out->shorts = min_len < glen + s.S - 1 ? 1u : 0u;
            }
        }
    }
    if (!found) return false;

    out->H.assign(out->words, 0);
    const uint32_t glen = out->glen, gw = out->gw, nb = out->nb;
    const uint32_t width = packed ? 2u : 8u;
    // a string as the kernel sees it: symbols at `width` bits, first lowest
    const uint32_t gm = gw * width >= 32 ? GRAM_MUL : GRAM_MUL << (32 - gw * width);
    auto insert = [&](uint64_t x) {
        const uint32_t t = (uint32_t)x;
        uint32_t y = t * gm;
        if (gw == 5 && !packed) y += (uint32_t)(x >> 8) * WIN_MUL2;
        const uint32_t w = (uint32_t)(((uint64_t)y * out->words) >> 32);
        for (uint32_t b = 0; b < nb; b++)
            out->H[w] |= 1u << ((uint32_t)(x >> (width * win_off(packed, b))) & 31u);
    };
    const uint32_t vals = 1u << bps;
    for (const WinPat &p : pats)
        for (uint32_t o = 0; o < out->stride; o++) {
            const uint32_t known = p.len > o ? std::min(p.len - o, glen) : 0u;
            uint64_t x = 0;
            for (uint32_t i = 0; i < known; i++) x |= (uint64_t)p.p[o + i] << (width * i);
            // every value of the symbols past the pattern's end
            uint64_t n = 1;
            for (uint32_t i = known; i < glen; i++) n *= vals;
            for (uint64_t c = 0; c < n; c++) {
                uint64_t xx = x, r = c;
                for (uint32_t i = known; i < glen; i++) {
                    xx |= (r % vals) << (width * i);
                    r /= vals;
                }
                insert(xx);
            }
        }
    return true;
}

}  // namespace pfac
