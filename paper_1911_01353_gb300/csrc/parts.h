// How many templates one CTA of the filter takes (host only).
//
// The bank's groups fix its rows and, in reduced precision, where the 16-bit
// roundings fall; a CTA takes a whole group or one of equal parts of it.  Time
// is counted in steps, one template of one CTA; setting a CTA up costs `setup` of
// them, and `slots` CTAs run at a time.  The part length is the one whose
// CTAs finish first on an idle chip, given the templates of every group that this
// spectrum searches (a sub-grid or a template range holds the narrow groups whole
// and few templates of the others): the longest CTA bounds a short spectrum,
// whole waves a longer one.  12 261 templates, FP32: 2^13 bins on a plan for 2^22
// in whole groups of 1024, 24 CTAs, 4.0 ms, in parts 0.94; a request of 83 000 bins
// and |z| <= 50, |w| <= 600 on 27 391 templates 2.97 ms whole, 1.18 in parts
// (whole calls).
//
// A plan for several spectra runs them together, and there each extra CTA's setup
// is lost time: its items are cut to 32 templates or more while the setups add no
// more than 1/24 to the item's steps, those of a plan for one spectrum to 4 (fewer
// are setup only: one CTA takes 30.7 us for 4 templates, 21.5 for one) while they add
// no more than half.  Nothing but the bank's plan and the item itself enters, so
// that an item's statistics are added in the same order alone, in every batch, and
// by every plan on the bank.
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

namespace jerk {

constexpr int kTried = 8;
constexpr int kPartWaves = 24;       // an item is cut to at most this many waves of CTAs (or twice its whole groups)

// a group's share of one item: `ctas` CTAs (of segments) walk `count` templates
struct PartGroup {
    int64_t ctas;
    int count;
};

struct PartRule {
    int slots;                       // CTAs that run at a time
    int setup;                       // steps that setting one up takes
    int least;                       // templates of a part at least
    int cost;                        // added setups are at most 1 / cost of the steps (0: any)
};

inline PartRule part_rule(int slots, int setup, bool batched) {
    return batched ? PartRule{slots, setup, 32, 24} : PartRule{slots, setup, 4, 2};
}

inline int64_t parts_of(int count, int length) { return (count + length - 1) / length; }

// Steps until every CTA of an item has finished, taken in order by whichever SM is
// free first (equal ones at once: `at` holds when how many SMs are free).
inline int64_t finish_time(const std::vector<PartGroup> &item, int length, const PartRule &r) {
    struct Level {
        int64_t time, sms;
    };
    std::vector<Level> at{{0, r.slots}};
    for (const PartGroup &g : item) {
        const int64_t parts = parts_of(g.count, length);
        const int64_t base = g.count / parts, more = g.count % parts;
        for (int u = 0; u < 2; ++u) {
            const int64_t steps = base + (u == 0 ? 1 : 0) + r.setup;
            for (int64_t left = (u == 0 ? more : parts - more) * g.ctas; left > 0;) {
                const int64_t n = std::min(left, at[0].sms), end = at[0].time + steps;
                left -= n;
                at[0].sms -= n;
                if (at[0].sms == 0) at.erase(at.begin());
                size_t i = 0;
                while (i < at.size() && at[i].time < end) ++i;
                if (i < at.size() && at[i].time == end)
                    at[i].sms += n;
                else
                    at.insert(at.begin() + i, Level{end, n});
            }
        }
    }
    return at.back().time;
}

// Templates per CTA at most; group g is cut into parts_of(g.count, result) equal
// parts.  Lengths are ranked by an estimate (one wave: the longest CTA; more: the
// whole waves of it or the work per SM and half a CTA, whichever is less), and of
// the best kTried the one that finishes first is taken.  Where whole groups are
// more waves than parts may be, the estimate decides.
inline int part_length(const std::vector<PartGroup> &item, const PartRule &r) {
    int most = 1;
    int64_t whole = 0, steps = 0;
    for (const PartGroup &g : item) {
        most = std::max(most, g.count);
        whole += g.ctas;
        steps += g.ctas * (g.count + r.setup);
    }
    struct Choice {
        double cost;
        int length;
        int64_t ctas;
    };
    std::vector<Choice> best;
    for (int64_t parts = 1, length = most;; parts = parts_of(most, (int)length - 1)) {
        length = parts_of(most, (int)parts);
        int64_t n = 0, work = 0;
        for (const PartGroup &g : item) {
            const int64_t p = parts_of(g.count, (int)length);
            n += g.ctas * p;
            work += g.ctas * (g.count + r.setup * p);
        }
        if (parts > 1 && n > std::max<int64_t>((int64_t)kPartWaves * r.slots, 2 * whole)) break;
        if (parts > 1 && length < r.least) break;
        if (parts > 1 && r.cost > 0 && work > steps + steps / r.cost) break;
        const double one = (double)(length + r.setup);
        const double waves = (double)((n + r.slots - 1) / r.slots) * one;
        const double cost = n <= r.slots ? one : std::max(one, std::min(waves, (double)work / r.slots + 0.5 * one));
        best.push_back({cost, (int)length, n});
        if (length == 1) break;
    }
    // (stable: of equal costs the longer part, listed first, stays first)
    std::stable_sort(best.begin(), best.end(), [](const Choice &a, const Choice &b) { return a.cost < b.cost; });
    if (best[0].ctas > (int64_t)kPartWaves * r.slots) return best[0].length;
    int length = 0;
    int64_t least = INT64_MAX;
    for (size_t i = 0; i < best.size() && i < kTried; ++i) {
        const int64_t t = finish_time(item, best[i].length, r);
        if (t < least || (t == least && best[i].length > length)) {
            least = t;
            length = best[i].length;
        }
    }
    return length;
}

// CTAs of any item whose whole groups are `whole` CTAs at most
inline int64_t part_ctas_bound(int64_t whole, const PartRule &r) {
    return std::max<int64_t>((int64_t)kPartWaves * r.slots, 2 * whole);
}

// ... and of `items` spectra together whose whole groups, of `most` templates or
// fewer, are `whole` CTAs at most: each item's own bound, or what the limit on the
// setups lets them come to
inline int64_t part_ctas_bound(int64_t whole, int64_t items, int most, const PartRule &r) {
    const int64_t each = items * kPartWaves * r.slots + 2 * whole;
    return r.cost > 0 ? std::min(each, whole + whole * (most + r.setup) / ((int64_t)r.cost * r.setup) + items) : each;
}

// launch-table entries of an item of `templates` templates in `groups` groups
inline int64_t part_entries_bound(int64_t groups, int64_t templates, const PartRule &r) {
    return groups + templates / r.least;
}

}  // namespace jerk
