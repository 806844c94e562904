// What the warp-segment kernels of rows with their own mesh (ram_nseg.cu, ram_nseg_f64.cu)
// take of a row: plan-time arithmetic on its nodes, host only (no CUDA).
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

namespace ram {

// A warp stages a window of kNsegWin source cells, kNsegHR of them on each side for the
// reconstructions' stencils, and takes segments of at most kNsegMost output cells,
// residual halo included.
constexpr int kNsegWin = 160;
constexpr int kNsegHR = 2;
constexpr int kNsegRoom = kNsegWin - 2 * kNsegHR;  // cells that edges may lie in
constexpr int kNsegMost = kNsegRoom - 4;
// the fewest of them that a row may use (see nseg_fit)
constexpr int kNsegLeast = 92;

struct NsegFit {
    int cells = 0;   // most cells of a segment with its halo; 0: left to the tiled kernels
    int window = 0;  // source cells of a window that edges may lie in
    int units = 0;   // the positions are in units of 2^units, see nseg_fit
};

// The most physical length of a window of c cells with its stencils' cells, and of the
// widest cell beyond.
inline double nseg_reach(const double *x, int n, double w_max, int c)
{
    const double L = x[n] - x[0];
    const int span = c + 2 * kNsegHR + 2;
    if (n <= span) return 2.0 * L;
    double len = 0.0;
    for (int st = 0; st < n; ++st)
        len = std::max(len, st + span <= n ? x[st + span] - x[st] : x[st + span - n] - x[st] + L);
    return len + w_max;
}

// Whether some interval as long as the widest cell touches more than `most` cells.
inline bool nseg_crowded(const double *w, int n, double w_min, double w_max, int most)
{
    if (w_max <= w_min * most) return false;
    int e = 0;
    double len = 0.0;  // of cells st .. e - 1 (cyclic)
    for (int st = 0; st < n; ++st) {
        while (e < st + n && len + w[e % n] < w_max) len += w[e++ % n];
        if (e - st + 2 > most) return true;
        if (e > st)
            len -= w[st];
        else
            e = st + 1;
    }
    return false;
}

// Most cells of a segment, halo included, for windows of c cells.  A segment whose source
// cells do not fit one window costs another window, so the length is the one with the
// least expected cost per output cell, windows over output cells, on 64 sampled
// placements (against the longest whose sampled placements all fit one window: 49.9 and
// 51.0 us on the 512-row batch of widths within [1/2, 2] x mean, 27.7 and 44.1 for the
// split step of 510 rings of 1533 cells on the bump mesh).
inline int nseg_cells(const double *x, int n, int c)
{
    const double L = x[n] - x[0];
    int best = 0;
    double cost = 1e300;
    for (int ne = std::min(kNsegMost, c - 4); ne >= 64; ne -= 8) {
        const int s = std::min(ne, n - 1);
        double windows = 0.0;
        for (int k = 0; k < 64; ++k) {
            const int i = (int)((2654435761ull * (2 * k + 1)) % (uint64_t)n);
            const int j = (int)((40503ull * 65537ull * (2 * k + 1) + n / 3) % (uint64_t)n);
            double len = (i + s <= n ? x[i + s] - x[i] : x[i + s - n] - x[i] + L) + x[j];
            int turn = 0;
            if (len > x[n]) {
                len -= L;
                turn = n;
            }
            const int e = (int)(std::upper_bound(x, x + n + 1, len) - x) + turn;
            windows += std::max(1, (e - j + c - 2) / (c - 1));
        }
        if (windows / (s - 4) < cost) {
            cost = windows / (s - 4);
            best = s;
        }
    }
    return best;
}

// What the FP32 (fit[0]) and the FP64 kernel (fit[1]) take of a row.  x: nodes, w: widths,
// n >= least cells (a segment of one cell with the widest residual halo spans less than a
// period).
//
// FP64: positions are the plan's 64-bit fractions of the period; rows about as long as a
// window or shorter take half of that resolution (units = 1), so that two turns fit 64
// bits.  Every cell is at least 2^20 of them.
//
// FP32: positions are 32-bit, in units of 2^units of the 64-bit fraction, and those of a
// window and of the edges over it span less than 2^32 units (the reach); rows not much
// longer than that take half the period's units (33).  Every cell keeps at least 2^20
// units.  A power of two, the unit doubles wherever the reach crosses one: on a 16:1 mesh
// the narrow cells would fall below 2^20 for a third of an octave of row lengths (512,
// 1024, 2048 and 4096 cells of the paper's bump mesh among them).  There the window is
// used only in part, as many cells as fit the finer unit: half of a full one at the worst
// where wide cells fill it, but for kNsegLeast.
//
// In both, one output cell lies over fewer source cells than the window holds.
inline void nseg_fit(const double *x, const double *w, int n, int least, NsegFit fit[2])
{
    fit[0] = fit[1] = NsegFit();
    if (n < least) return;
    const double L = x[n] - x[0];
    if (!(L > 1e-250 && L < 1e250)) return;  // widths are scaled by their exponents
    const double two64 = 18446744073709551616.0, least_units = 1048576.0;
    double w_min = w[0], w_max = w[0];
    for (int i = 1; i < n; ++i) {
        w_min = std::min(w_min, w[i]);
        w_max = std::max(w_max, w[i]);
    }
    const double narrow = w_min / L * two64;  // of the 64-bit fraction
    if (narrow < least_units) return;
    auto units = [&](int c) {
        const double reach = nseg_reach(x, n, w_max, c);
        if (reach > 0.999 * L) return 33;
        return std::max(0, (int)std::ceil(std::log2(reach / L * two64 * 1.000001)) - 32);
    };
    auto fine = [&](int u) { return std::ldexp(narrow, -u) >= least_units; };
    const int u = units(kNsegRoom);
    if (!nseg_crowded(w, n, w_min, w_max, kNsegRoom - 8))
        fit[1] = NsegFit{nseg_cells(x, n, kNsegRoom), kNsegRoom, u > 32 ? 1 : 0};
    if (fine(u)) {
        if (fit[1].cells) fit[0] = NsegFit{fit[1].cells, kNsegRoom, u};
        return;
    }
    // the most cells whose unit is fine enough (the reach grows with them)
    int lo = kNsegLeast, hi = kNsegRoom;
    if (!fine(units(lo))) return;
    while (hi - lo > 1) {
        const int mid = (lo + hi) / 2;
        (fine(units(mid)) ? lo : hi) = mid;
    }
    if (!nseg_crowded(w, n, w_min, w_max, lo - 8))
        fit[0] = NsegFit{nseg_cells(x, n, lo), lo, units(lo)};
}

}  // namespace ram
