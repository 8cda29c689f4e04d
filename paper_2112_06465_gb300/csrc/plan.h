// plan.h -- decisions of the host side that need no device: which matrices get
// the row-per-lane layout,
// which products read it, how a solve runs and how a sweep shares the SMs.  Plain
// C++, so that a test compiles it by itself.
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

namespace hz {

constexpr int kSlMaxWidth = 64;    // steps per slice at most (bits of the mask)
constexpr int kSlMaxRow = 512;     // entries of a long row at most
// A row longer than this many entries and twice the mean leaves its slots
// empty and is summed by all lanes of its slice's warp from the CSR arrays:
// one such row in a slice would make every lane step through its length.
// (618 k rows of 15, 161 of them 97 to 195 long: 115 us a product that way, 52
// us this way, 60 us as lane runs.)
constexpr int kSlLongRow = 32;
constexpr int kSlLongG = 8;        // loads of such a row in flight per lane: 256 entries a pass
// The warp takes its long rows one after the other, so long rows that lie
// together keep one warp busy while the others have finished: at most this
// many passes over all long rows of a slice.  us a product from cold caches,
// 20 k rows of 15 with some of 400 side by side (lane runs 15.0, without long
// rows 10.9), four loads in flight: 1 row 17, 2 rows 23, 8 rows 62, 32 rows
// 165, and a BiCGStab iteration with 32 of them 261 against the graph's 53;
// eight in flight: 1 row 15, 2 rows of 255 17.
constexpr int kSlLongPasses = 2;

// The row-per-lane layout of a CSR pattern: slices of 32 rows, one per lane,
// as wide as the slice's longest row that is not a long one.
struct SlicePlan {
    bool fits = false;
    std::vector<int32_t> base;     // [slices + 1] first step of each slice
    std::vector<unsigned> longs;   // [slices] lanes of long rows
    int64_t slots = 0;
    int64_t nlong = 0;
    int32_t most = 0;              // entries of the fullest slice
    int32_t width = 0;             // steps of the widest slice
};

// Padded rows cost binary64 instructions, so the padded size may exceed the
// entries by a quarter (the lane-run stream's row switches and second
// accumulator cost it 26 % more binary64 instructions than the multiply-adds
// it needs: 728 k against 577 k on 618 k rows of 15), by two fifths where the
// work is small and launches and latency count instead: rows of 9 to 17 in
// random order, padded by 1.3, lane runs / slices, a product 9.0 / 5.6 us at
// 4,000 rows and 15.1 / 8.2 at 64,000, a BiCGStab iteration 54 / 25 and 78 /
// 42.
inline SlicePlan slice_plan(const int32_t *rp, int32_t n, int32_t nnz) {
    SlicePlan p;
    if (n <= 0 || nnz <= 0) return p;
    const int ns = (n + 31) / 32;
    p.base.resize(ns + 1);
    p.longs.assign(ns, 0u);
    const double lim = std::max((double)kSlLongRow, 2.0 * ((double)nnz / n));
    int64_t P = 0, short_nnz = nnz;
    int rmax = 0, passes_max = 0;
    for (int q = 0; q < ns; ++q) {
        const int r0 = 32 * q, r1 = std::min(n, r0 + 32);
        int w = 0, passes = 0;
        const int32_t *row = rp + r0;
        if (r1 - r0 == 32)   // (a loop that vectorises: every row of every new operator passes here)
            for (int r = 0; r < 32; ++r) w = std::max(w, row[r + 1] - row[r]);
        else
            for (int r = 0; r < r1 - r0; ++r) w = std::max(w, row[r + 1] - row[r]);
        rmax = std::max(rmax, w);
        if (w > lim) {
            w = 0;
            for (int r = r0; r < r1; ++r) {
                const int len = rp[r + 1] - rp[r];
                if (len > lim) {
                    p.longs[q] |= 1u << (r & 31);
                    p.nlong += 1;
                    short_nnz -= len;
                    passes += (len + 32 * kSlLongG - 1) / (32 * kSlLongG);
                } else {
                    w = std::max(w, len);
                }
            }
        }
        p.base[q] = (int32_t)std::min<int64_t>(P, INT32_MAX);
        p.most = std::max(p.most, rp[std::min(n, 32 * q + 32)] - rp[32 * q]);
        P += w;
        p.width = std::max(p.width, w);
        passes_max = std::max(passes_max, passes);
    }
    p.base[ns] = (int32_t)std::min<int64_t>(P, INT32_MAX);
    p.slots = 32 * P;
    p.fits = P > 0 && p.width <= kSlMaxWidth && rmax <= kSlMaxRow && 128 * p.nlong <= n && passes_max <= kSlLongPasses &&
             p.slots < INT32_MAX - 32 &&
             (4 * p.slots <= 5 * short_nnz || (n <= 65536 && 5 * p.slots <= 7 * short_nnz));
    return p;
}

// Whether a product by itself reads the slices (the solves on chip always do).
// A slice is one warp's serial walk over its width, so where there are few of
// them and they are wide, the row blocks, which spread every row over a warp's
// lanes, are faster: binary64 on the caller's arrays, complex64 on its copy.
// us a product, warm, row blocks / slices:
//   rows of           60          40          27      30 to 60
//   binary64
//     4,000       6.6 / 11.7   6.7 / 8.9  10.3 / 7.0   9.1 / 12.1
//    10,000       9.6 / 12.7   9.2 / 8.9  10.5 / 7.2  11.5 / 12.6
//    14,000      10.1 / 12.9       - / 9.1     - / 7.0  14.4 / 12.8
//    24,000      16.8 / 13.9  13.9 / 9.8  16.1 / 7.9  17.9 / 14.0
//   complex64
//     4,000       5.4 / 6.7    5.5 / 5.3   5.1 / 4.7   5.8 / 7.1
//    24,000       6.6 / 8.2    6.5 / 5.8   5.7 / 5.1   6.6 / 8.2
//    64,000      12.2 / 10.5  12.2 / 7.6   6.6 / 6.0  11.7 / 10.4
inline bool slice_product(int nsl, int width, bool binary64, int num_sms) {
    if (binary64) return !((width >= 40 && 2 * nsl <= 3 * num_sms) || (width > 52 && 2 * nsl <= 5 * num_sms));
    return !(width > 40 && nsl <= 5 * num_sms);
}

// How a solve runs, and what it falls back to where the device has no room for
// a launch (a partition, or a share of the SMs given to other work): one
// cluster, every SM, the graph of kernels.
enum class Way { cluster, all_sms, graph };
enum class Launch { done, no_room, error };
// launch(way) on the ways from `way` on until one is taken; the graph is the
// caller's.  True unless a launch failed for another reason.
template <class F> inline bool first_way(Way &way, F launch) {
    while (way != Way::graph) {
        const Launch r = launch(way);
        if (r != Launch::no_room) return r == Launch::done;
        way = way == Way::cluster ? Way::all_sms : Way::graph;
    }
    return true;
}

// The CTAs of each system of a sweep on chip, one CTA per SM: nsl slices each
// (0: an empty system, no CTA), at most max_cta CTAs a system and max_slices
// slices a CTA.  Shares by slices, then one CTA more at a time to the system
// whose CTAs own the most; where rounding the small shares up to one CTA and
// the others down leaves too few, every system starts from one.  False where
// they do not fit.
// us per iteration of the slowest system, in the grid-wide phases / on chip,
// all systems running (rows of 7, 15 and 27 entries):
//   64,000 unknowns with 100 boxes of 1,000    146 / 58   179 / 84   259 / 116
//   125,000 unknowns with 80 boxes of 1,000    146 / 66   182 / 104  263 / 151
inline bool sweep_plan(const std::vector<int> &nsl, int num_sms, int max_cta, int max_slices, std::vector<int> *ncta) {
    const int ns = (int)nsl.size();
    std::vector<int> &c = *ncta;
    int64_t total = 0;
    int live = 0;
    for (int n : nsl) {
        total += n;
        live += n > 0;
    }
    c.assign(ns, 0);
    if (live > num_sms) return false;
    auto cap = [&](int k) { return std::min(nsl[k], max_cta); };
    for (int start = 0; start < 2; ++start) {
        int left = num_sms;
        for (int k = 0; k < ns; ++k) {
            if (nsl[k] == 0) continue;
            c[k] = start ? 1 : std::max(1, std::min(cap(k), (int)((int64_t)num_sms * nsl[k] / total)));
            left -= c[k];
        }
        if (left < 0) continue;
        for (; left > 0; --left) {
            int best = -1;
            double most = 0.0;
            for (int k = 0; k < ns; ++k) {
                if (c[k] == 0 || c[k] >= cap(k)) continue;
                const double load = (double)nsl[k] / c[k];
                if (load > most) { most = load; best = k; }
            }
            if (best < 0) break;
            c[best] += 1;
        }
        bool ok = true;
        for (int k = 0; k < ns; ++k) ok = ok && (c[k] == 0 || (nsl[k] + c[k] - 1) / c[k] <= max_slices);
        if (ok) return true;
    }
    return false;
}

}  // namespace hz
