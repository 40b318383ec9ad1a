// Host construction of the work lists of the tensor-core far field: groups of G consecutive
// target blocks share one MMA (N = G x 64 targets), so each group walks the union of its
// blocks' lists with a mask per entry of the blocks that own it.  Plain C++ (no CUDA types):
// the test suite compiles this header with the host compiler.
#pragma once
#include <algorithm>
#include <cstdint>
#include <cstdlib>
#include <utility>
#include <vector>

namespace lspr {

struct TcEntry {   // layout of int2
    int box, mask;
};
struct TcItem {    // layout of int4
    int group, begin, end, pad;
};
struct TcRange {   // layout of int4
    int s0, s1, mask, pad;
};

// The size of the units when `total` boxes or sources are spread over `sms` persistent blocks: as
// long as some 2.5 units per block remain, between lo and hi.  M2P of 20480 panels, 16 right-hand sides
// (23979 boxes, 152 blocks): 268, 240, 279 us with units of 32, 64, 128 boxes; 81920 panels, 64 (80757
// boxes): 1574, 1470, 1419 us, where the error sets the limit (lspr_internal.cuh).
inline int tc_unit(int64_t total, int sms, int lo, int hi) {
    const int64_t n = 2 * total / (5 * (int64_t)std::max(1, sms));
    return (int)std::min<int64_t>(hi, std::max<int64_t>(lo, n));
}

// M2P: per group of G consecutive target blocks, the union of the blocks' box lists sorted by
// box, each box with the mask of the blocks whose list holds it, as one unit.  items:
// [nitems][4] = (block, list begin, list end, -) into list (box ids); a block's items cover its list.
inline void tc_union_m2p(int64_t nblocks, int G, const int *list, const int *items, int64_t nitems,
                         std::vector<TcEntry> &out, std::vector<TcItem> &units) {
    out.clear();
    units.clear();
    const int64_t ngroups = (nblocks + G - 1) / G;
    std::vector<std::vector<TcEntry>> per((size_t)ngroups);
    for (int64_t i = 0; i < nitems; ++i) {
        const int *it = items + 4 * i;
        const int64_t g = it[0] / G;
        const int bit = 1 << (it[0] % G);
        for (int l = it[1]; l < it[2]; ++l) per[g].push_back(TcEntry{list[l], bit});
    }
    for (int64_t g = 0; g < ngroups; ++g) {
        std::vector<TcEntry> &v = per[g];
        if (v.empty()) continue;
        std::sort(v.begin(), v.end(), [](const TcEntry &a, const TcEntry &b) { return a.box < b.box; });
        const int64_t start = (int64_t)out.size();
        for (const TcEntry &e : v) {
            if ((int64_t)out.size() > start && out.back().box == e.box)
                out.back().mask |= e.mask;
            else
                out.push_back(e);
        }
        units.push_back(TcItem{(int)g, (int)start, (int)out.size(), 0});
    }
}

// the units of tc_union_m2p cut into units of at most seg boxes of nearly equal size
inline void tc_cut_m2p(int seg, std::vector<TcItem> &units) {
    std::vector<TcItem> cut;
    for (const TcItem &u : units) {
        const int64_t n = u.end - u.begin, k = (n + seg - 1) / seg;
        for (int64_t q = 0; q < k; ++q)
            cut.push_back(TcItem{u.group, (int)(u.begin + n * q / k), (int)(u.begin + n * (q + 1) / k), 0});
    }
    units.swap(cut);
}

inline void tc_group_m2p(int64_t nblocks, int G, int seg, const int *list, const int *items, int64_t nitems,
                         std::vector<TcEntry> &out, std::vector<TcItem> &units) {
    tc_union_m2p(nblocks, G, list, items, nitems, out, units);
    tc_cut_m2p(seg, units);
}

// P2P: per group, the blocks' source ranges are cut at every range end (a sweep over the sorted
// ends with one coverage count per block); pieces with the same mask that touch are merged, and
// a group's pieces are one unit.  items: [nitems][4] = (block, source begin, source end, -); the
// ranges of one block do not overlap.  Returns the number of sources over all pieces.
inline int64_t tc_union_p2p(int64_t nblocks, int G, const int *items, int64_t nitems, std::vector<TcRange> &out,
                            std::vector<TcItem> &units) {
    out.clear();
    units.clear();
    int64_t total = 0;
    const int64_t ngroups = (nblocks + G - 1) / G;
    std::vector<std::vector<std::pair<int, int>>> ev((size_t)ngroups);   // (position, +-(block + 1))
    for (int64_t i = 0; i < nitems; ++i) {
        const int *it = items + 4 * i;
        if (it[2] <= it[1]) continue;
        const int64_t g = it[0] / G;
        const int k = it[0] % G + 1;
        ev[g].push_back({it[1], k});
        ev[g].push_back({it[2], -k});
    }
    std::vector<int> cov((size_t)G);
    for (int64_t g = 0; g < ngroups; ++g) {
        std::vector<std::pair<int, int>> &e = ev[g];
        if (e.empty()) continue;
        std::sort(e.begin(), e.end(), [](const std::pair<int, int> &a, const std::pair<int, int> &b) {
            return a.first < b.first;
        });
        std::fill(cov.begin(), cov.end(), 0);
        const size_t first = out.size();
        for (size_t i = 0; i < e.size();) {
            const int pos = e[i].first;
            for (; i < e.size() && e[i].first == pos; ++i) cov[std::abs(e[i].second) - 1] += e[i].second > 0 ? 1 : -1;
            if (i == e.size()) break;
            int mask = 0;
            for (int k = 0; k < G; ++k) mask |= cov[k] > 0 ? 1 << k : 0;
            const int next = e[i].first;
            if (!mask) continue;
            if (out.size() > first && out.back().s1 == pos && out.back().mask == mask)
                out.back().s1 = next;
            else
                out.push_back(TcRange{pos, next, mask, 0});
        }
        for (size_t q = first; q < out.size(); ++q) total += out[q].s1 - out[q].s0;
        if (out.size() > first) units.push_back(TcItem{(int)g, (int)first, (int)out.size(), 0});
    }
    return total;
}

// the units of tc_union_p2p cut: pieces longer than seg_src are split, and consecutive pieces are packed
// into units of at most seg_src sources
inline void tc_cut_p2p(int seg_src, std::vector<TcRange> &pieces, std::vector<TcItem> &units) {
    std::vector<TcRange> out;
    std::vector<TcItem> cut;
    for (const TcItem &u : units) {
        int u0 = (int)out.size(), usrc = 0;
        for (int q = u.begin; q < u.end; ++q) {
            const TcRange &p = pieces[q];
            for (int s0 = p.s0; s0 < p.s1;) {
                const int n = std::min(p.s1 - s0, seg_src);
                if (usrc > 0 && usrc + n > seg_src) {
                    cut.push_back(TcItem{u.group, u0, (int)out.size(), 0});
                    u0 = (int)out.size();
                    usrc = 0;
                }
                out.push_back(TcRange{s0, s0 + n, p.mask, 0});
                usrc += n;
                s0 += n;
            }
        }
        if ((int)out.size() > u0) cut.push_back(TcItem{u.group, u0, (int)out.size(), 0});
    }
    pieces.swap(out);
    units.swap(cut);
}

inline int64_t tc_group_p2p(int64_t nblocks, int G, int seg_src, const int *items, int64_t nitems,
                            std::vector<TcRange> &out, std::vector<TcItem> &units) {
    const int64_t total = tc_union_p2p(nblocks, G, items, nitems, out, units);
    tc_cut_p2p(seg_src, out, units);
    return total;
}

}  // namespace lspr
