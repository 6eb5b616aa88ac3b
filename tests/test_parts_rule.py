"""How the filter's template groups are cut over CTAs (csrc/parts.h, compiled for
the host): short spectra on a plan for long ones, sub-grids of a large bank at
any length, template ranges.  The chosen part length must finish, taken in order
by 152 SMs, within a tenth of the best length of 4 templates or more; on a shared plan no later
than whole groups of two-segment CTAs at their shorter step (2.4 against 3.0 us),
with no more than 1/24 of setups added; and its CTAs and launch-table entries must
stay within the bounds that size a plan's workspace."""
import heapq
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1911_01353_gb300", "csrc")
SMS, SETUP, L = 152, 5, 4096

MAIN = r"""
#include <cstdio>
#include "parts.h"
using namespace jerk;
int main() {
    int shared, items, groups, most;
    long long templates;
    while (std::scanf("%d %d %d %lld", &shared, &items, &groups, &templates) == 4) {
        const PartRule r = part_rule(152, 5, shared != 0);
        std::vector<PartGroup> item(groups);
        int64_t whole = 0;
        most = 1;
        for (auto &g : item) {
            long long c;
            std::scanf("%lld %d", &c, &g.count);
            g.ctas = c;
            whole += c;
            most = std::max(most, g.count);
        }
        const int len = part_length(item, r);
        std::printf("%d %lld %lld %lld %lld\n", len, (long long)finish_time(item, len, r),
                    (long long)part_ctas_bound(whole, r), (long long)part_ctas_bound(whole * items, items, most, r),
                    (long long)part_entries_bound(groups, templates, r));
    }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("parts")
    (d / "main.cc").write_text(MAIN)
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-I", CSRC, str(d / "main.cc"), "-o", str(d / "main")])

    def ask(queries):
        """(shared, items of the plan, [(ctas, count)]) -> (length, finish, bound of one, bound of all, entries)"""
        text = "".join("%d %d %d %d %s\n" % (s, k, len(it), sum(c for _, c in it), " ".join("%d %d" % g for g in it))
                       for s, k, it in queries)
        out = subprocess.run([str(d / "main")], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    return ask


class Bank:
    """Groups of a bank as a plan for max_bins bins orders them."""

    def __init__(self, zmax, wmax, max_bins, size=0):
        z, w = np.meshgrid(np.arange(-zmax, zmax + 1, 2), np.arange(-wmax, wmax + 1, 20))
        self.z, self.w = z.ravel(), w.ravel()
        m = (4 * abs(self.z) + abs(self.w) + 7) // 8 + 16
        T = m.size
        nseg = -(-2 * max_bins // (L - 4 * m.max()))
        size = min(size or min(max(-(-T * nseg // (6 * SMS)), 8), 1024), T)
        order = np.argsort(m, kind="stable")
        self.groups = [(np.sort(order[k:k + size]), L - 4 * m[order[k:k + size]].max()) for k in range(0, T, size)]

    def item(self, n, zs=None, ws=None, lo=None, hi=None, segs=3):
        out = []
        for t, V in self.groups:
            if zs is not None:
                t = t[(abs(self.z[t]) <= zs) & (abs(self.w[t]) <= ws)]
            if lo is not None:
                t = t[(t >= lo) & (t < hi)]
            if t.size:
                out.append((-(-(-(-2 * n // V)) // segs), int(t.size)))
        return out


def parts(count, length):
    p = -(-count // length)
    return [count // p + (1 if i < count % p else 0) for i in range(p)]


def finish(item, length):
    free = [0] * SMS
    for ctas, count in item:
        for steps in parts(count, length):
            for _ in range(ctas):
                heapq.heapreplace(free, free[0] + steps + SETUP)
    return max(free)


def ctas(item, length):
    return sum(c * len(parts(k, length)) for c, k in item)


LENGTHS = (50000, 54000, 57000, 60000, 83000, 100000, 113000, 116000, 141000, 171000)


def test_alone_finishes_near_the_best(rule):
    big = Bank(200, 600, 1 << 22)
    items = [big.item(n) for n in (1, 3000, 1 << 13, 1 << 14, 1 << 15, 1 << 16)]
    items += [big.item(n, lo=3000, hi=5000) for n in (1 << 13, 1 << 15)] + [big.item(1 << 14, lo=77, hi=78)]
    large = Bank(300, 900, 1 << 22)
    items += [large.item(n, 50, 600) for n in LENGTHS[::3]] + [large.item(n, 300, 0) for n in LENGTHS[::4]]
    items += [Bank(20, 60, 1 << 16).item(n) for n in (1 << 13, 1 << 16)]
    items += [Bank(40, 300, 40000, size=300).item(n) for n in (5000, 40000)]
    for item, (length, end, bound, _, entries) in zip(items, rule([(0, 1, it) for it in items])):
        tried = [1 << 20] + sorted({-(-k // q) for _, k in item for q in range(1, k + 1) if -(-k // q) >= 4})
        best = min(finish(item, c) for c in tried if ctas(item, c) <= bound)
        assert end == finish(item, length)
        assert end <= 1.1 * best, (item, length, end, best)
        assert ctas(item, length) <= bound and sum(len(parts(k, length)) for _, k in item) <= entries


def test_shared_plan_is_no_slower_than_whole_groups(rule):
    bank = Bank(300, 900, 1 << 22)
    cases = [(n, z, w) for n in LENGTHS for z, w in ((50, 600), (100, 300), (300, 0), (200, 300))]
    items = [bank.item(*c) for c in cases]
    for c, item, (length, end, bound, both, entries) in zip(cases, items, rule([(1, 8, it) for it in items])):
        before = 2.4 * finish(bank.item(*c, segs=2), 1 << 20)
        assert 3.0 * end <= 1.02 * before, (c, length, end, before)
        steps = [sum(k * (q + SETUP) for k, m in item for q in parts(m, x)) for x in (length, 1 << 20)]
        assert steps[0] <= steps[1] * (1 + 1 / 24)
        assert ctas(item, length) <= bound and 8 * ctas(item, length) <= both
        assert sum(len(parts(k, length)) for _, k in item) <= entries


def test_short_groups_of_a_shared_plan_stay_whole(rule):
    items = [Bank(20, 60, 600000).item(n) for n in (1 << 13, 40000)]
    assert all(length >= 32 for length, *_ in rule([(1, 24, it) for it in items]))


def test_partials_of_a_server_plan(rule):
    # 27 391 templates, 2^24 bins in up to 32 spectra: all groups cut into as many parts
    # as one of 1024 can be, twice over, were 98 MB of partials
    bank = Bank(300, 900, 1 << 24)
    one = [((c + 31) // 32 + 1, k) for c, k in bank.item(1 << 24)]
    both = rule([(1, 32, one)])[0][3]
    assert 16 * both < 12e6
