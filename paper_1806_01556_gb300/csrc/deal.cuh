// How the convolution's work is dealt out to CTAs and worker groups. Plain integer code, the same on the host
// and on the device.
#pragma once
#include <numeric>

#include "fdas_internal.cuh"

namespace fdas {
namespace {

__host__ __device__ constexpr int lesser(int a, int b) { return a < b ? a : b; }
__host__ __device__ constexpr int greater(int a, int b) { return a > b ? a : b; }

// How the work, every segment with every template, is dealt out to the workers (CTAs, or worker groups of
// the tensor-core form). An item is a run of templates of one segment; its segment is transformed once.
//   per_seg > 0  shares: the segments lie one after the other on a line, each `lead` units for its forward
//                transform and then its templates, `unit` of them per unit of length; worker x takes the
//                x-th of n_workers equal pieces of the line.
//   per_seg = 0  chunks of t_chunk templates, n_tchunk per segment, dealt out round robin.
// The FP32 form numbers the templates of a segment in an order that takes neighbours apart (place t is template
// t stride mod n_temp), so that the rows around a strong signal, which all cross their thresholds at the same
// columns, fall to different workers: a search at 65536 bins with tones takes 38 us, 43 us in the plain order.
// The tensor-core form does the same with its pairs, with shares and HP_1.
struct Deal {
    int n_seg;  // of all spectra
    int n_temp;
    int per_seg, lead, unit;
    int n_workers;
    int t_chunk, n_tchunk;
    int stride;
};
// Worker x's first item (q < 0), or the one after the item that ended with place t1 of segment q: segment q (of
// all spectra) with places [t0, t1). False after the last. Nothing but q and t1, which the item needs anyway, is
// kept from one item to the next: more live values cost the FP32 convolution with HP_1 2% (402 us against 394 us
// at 2^21 bins). n_running: workers that run (chunks).
__host__ __device__ inline bool deal_next(const Deal &d, int x, int n_running, int &q, int &t0, int &t1) {
    if (d.per_seg == 0) {
        const int item = q < 0 ? x : q * d.n_tchunk + (t1 - 1) / d.t_chunk + n_running;
        if (item >= d.n_seg * d.n_tchunk) return false;
        q = item / d.n_tchunk;
        t0 = (item - q * d.n_tchunk) * d.t_chunk;
        t1 = lesser(t0 + d.t_chunk, d.n_temp);
        return true;
    }
    if (x >= d.n_workers) return false;
    const long long len = (long long)d.n_seg * d.per_seg;
    const int end = (int)(len * (x + 1) / d.n_workers);
    int pos = q < 0 ? (int)(len * x / d.n_workers) : t1 == d.n_temp ? (q + 1) * d.per_seg : end;
    while (pos < end) {
        q = pos / d.per_seg;
        const int from = pos - q * d.per_seg, to = lesser(d.per_seg, from + (end - pos));
        pos += to - from;
        t0 = greater(0, from - d.lead) * d.unit;
        t1 = lesser(greater(0, to - d.lead) * d.unit, d.n_temp);
        if (t0 < t1) return true;  // a piece that ends inside a segment's lead leaves the segment to the next worker
    }
    return false;
}

// Worker number of group g (of `groups`) of CTA `block` (of `grid`). Shares, and chunks that leave every CTA a group
// without work, go to different CTAs, and so to different SMs, before any CTA gets a second one: one or two groups
// alone on an SM run faster than three (BF16X3 convolution of 9768 bins 22.9 -> 18.6 us, 26048 bins 33.2 -> 24.8,
// 65536 bins in items of 43 templates 90 -> 56). With more chunks some SM has a full set of groups anyway, and chunks
// that are neighbours in one CTA read different templates, where workers that share one at the same time slow one
// another (54000 bins, 127 rows: 33.5 us, 34.5 us spread out).
__host__ __device__ inline int worker(const Deal &d, int block, int grid, int g, int groups) {
    const bool spread = d.per_seg > 0 || d.n_seg * d.n_tchunk <= grid * (groups - 1);
    return spread ? block + grid * g : block * groups + g;
}

// Chunks of templates_per_item templates, or (0) shares for up to per_sm (1 to 3) workers on each of `sms`
// SMs. *workers: how many workers have something to do.
//
// Shares keep every place of the GPU busy to the end at any length: one item per segment leaves a spectrum
// of 4099 bins on 3 of 152 SMs, and items of equal size end in a partial round. A worker pays one forward
// transform more than it owns, when its piece starts inside a segment. Three workers run on an SM; with
// little to do, fewer are faster, because one or two alone run faster than three: the number k per SM
// minimises (length of a piece + one transform + half a place for a second item's setup) x (time per place
// with k on an SM, relative to three). Equal items, one per worker and so without the second setup, are taken
// where they come out lower (short spectra). The leads and factors are fitted to timings from 4099 to 2^21
// bins. Convolution in us with one item per segment (44 templates per item in the tensor-core form), with the
// best equal items, and with this rule:
//   FP32    4099 bins 72, 13, 12   200003 bins 73, 51, 45   524288 bins 139, 111, 102
//           1000003 bins 226, 203, 185   2^21 bins 393, 380, 378   4194303 bins, 257 taps 686, 678, 677
//   BF16X3  200003 bins 74, 66, 63   1000003 bins 253, 250, 230   2^21 bins 489, 488, 429
inline Deal make_deal(const Geometry &g, int n_seg, int templates_per_item, int sms, int per_sm, int *workers) {
    Deal d{};
    d.n_seg = n_seg;
    d.n_temp = g.n_temp;
    const bool fp32 = g.precision == FDAS_FP32;
    d.unit = fp32 ? 1 : 2;
    const int units = (g.n_temp + d.unit - 1) / d.unit;  // of a segment
    // The stride nearest above the golden section of the units without a common factor.
    d.stride = (int)(0.618 * units) + 1;
    while (std::gcd(d.stride, units) != 1) ++d.stride;
    d.stride %= units;
    auto items = [&](int t_chunk) {
        d.per_seg = 0;
        d.t_chunk = t_chunk < g.n_temp ? t_chunk : g.n_temp;
        d.n_tchunk = (g.n_temp + d.t_chunk - 1) / d.t_chunk;
        *workers = n_seg * d.n_tchunk;
    };
    if (templates_per_item > 0) {
        items(templates_per_item);
        return d;
    }
    d.lead = fp32 ? 3 : 2;
    d.per_seg = units + d.lead;
    const long long len = (long long)n_seg * d.per_seg;
    const double start = fp32 ? 2.5 : 2.0, again = 0.5;
    const double pace[3] = {fp32 ? 0.54 : 0.49, fp32 ? 0.77 : 0.79, 1.0};
    double best = 0.0, best_whole = 0.0;
    int whole = 0;  // units per item when every worker takes one item
    for (int k = 1; k <= per_sm; ++k) {
        const long long most = (long long)n_seg * units;
        const int w = (int)(most < (long long)k * sms ? most : (long long)k * sms);
        const double cost = ((double)len / w + start + again) * pace[k - 1];
        if (k == 1 || cost < best) {
            best = cost;
            d.n_workers = w;
        }
        const int m = k * sms / n_seg < units ? k * sms / n_seg : units;  // items per segment
        if (m == 0) continue;
        const int u = (units + m - 1) / m;
        const double c = (u + start) * pace[k - 1];
        if (whole == 0 || c < best_whole) {
            best_whole = c;
            whole = u;
        }
    }
    if (whole > 0 && best_whole <= best) {
        items(whole * d.unit);
        return d;
    }
    *workers = d.n_workers;
    return d;
}

}  // namespace
}  // namespace fdas
