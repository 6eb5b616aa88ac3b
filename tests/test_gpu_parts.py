"""Template groups cut into parts over CTAs, bit for bit against plane rows: the
whole bank, a sub-grid, a template range and ranges of plane rows of a spectrum
whose groups of 300 are cut, and CTAs that walk 256, 512 and more templates (the
8-bit argmax is flushed every 256 of a group of warps) where whole groups just
fill the chip.  Every max-projection is the maximum of the rows the same plan
computes for the whole plane; FP32 names the lowest template that reaches it, the
16-bit filter one that reaches it (it compares powers before their scale)."""
import numpy as np
import pytest

import synth
from parity import lib_ready

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return lib_ready()


def check(plan, rows, ts, precision, item=0):
    """The stage-1 max-projection against the rows of the templates ts."""
    M, t = plan.maxproj(0, item=item)
    r = rows[torch.as_tensor(ts, device="cuda")] if len(ts) < rows.shape[0] else rows
    best = r.max(dim=0).values
    assert np.array_equal(M, best.cpu().numpy())
    cell = torch.arange(rows.shape[1], device="cuda")
    t = torch.from_numpy(t.astype(np.int64)).cuda()
    assert torch.equal(rows[t, cell], best)
    if precision == 0:
        first = torch.as_tensor(ts, device="cuda")[(r == best).to(torch.uint8).argmax(dim=0)]
        assert torch.equal(t, first)


def whole_plane(plan, x):
    rows = torch.empty(plan.info.n_templates, 2 * x.numel(), device="cuda")
    plan.plane(x, 0, rows.shape[0], rows)
    torch.cuda.synchronize()
    return rows


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("n,batch", [(5003, 1), (40001, 1), (90001, 2)])
def test_cut_groups(pkg, n, batch, precision):
    p = pkg.make_params(40, 2, 300, 20, stages=(1,), thresh=(1e9,), thresh_mode=pkg.THRESH_SIGMA, max_bins=2 * n,
                        group_size=300, precision=precision, max_batch=batch)
    x = torch.from_numpy(synth.spectrum(n, 95, [synth.Signal(n / 2.5, 20.0, 0.0, 30.0, 0.3)])).cuda()
    with pkg.Plan(p) as plan:
        T = plan.info.n_templates
        rows = whole_plane(plan, x)
        every = np.arange(T)
        z, w = 2 * (every % 41) - 40, 20 * (every // 41) - 300
        plan.search(x)
        plan.candidates()
        check(plan, rows, every, precision)
        mu, sd, _ = plan.stats()
        d = rows.double()
        assert mu[0] == pytest.approx(float(d.mean()), rel=1e-6)
        assert sd[0] == pytest.approx(float(d.std(unbiased=False)), rel=1e-6)
        del d
        for lo, hi in ((0, 1), (T - 1, T), (3, 700), (500, T)):
            plan.search_range(x, lo, hi)
            check(plan, rows, every[lo:hi], precision)
        grids = ((40, 0), (10, 300)) if batch == 2 else ((12, 160),)
        plan.search_batch([x] * len(grids), zmax=[g[0] for g in grids], wmax=[g[1] for g in grids], transient=True)
        plan.candidates()
        for i, (zm, wm) in enumerate(grids):
            check(plan, rows, every[(abs(z) <= zm) & (abs(w) <= wm)], precision, item=i)
        for t0, nt in ((0, 1), (T - 1, 1), (37, 300), (299, 2), (900, T - 900)):
            part = torch.empty(nt, 2 * n, device="cuda")
            plan.plane(x, t0, nt, part)
            torch.cuda.synchronize()
            assert torch.equal(part, rows[t0:t0 + nt])


# 595 templates, at most 3828 valid cells per segment: 50 and 75 CTAs for three groups
# and two, 150 for one group
@pytest.mark.parametrize("n,group_size,precision", [(287000, 256, 0), (430000, 298, 0), (861000, 595, 0),
                                                    (287000, 512, 2), (574000, 595, 2)])
def test_long_groups(pkg, n, group_size, precision):
    p = pkg.make_params(16, 2, 340, 20, stages=(1,), thresh=(1e9,), max_bins=n, group_size=group_size,
                        precision=precision)
    x = torch.from_numpy(synth.spectrum(n, 96)).cuda()
    with pkg.Plan(p) as plan:
        rows = whole_plane(plan, x)
        plan.search(x)
        plan.candidates()
        check(plan, rows, np.arange(plan.info.n_templates), precision)


@pytest.mark.parametrize("n", [5003, 40001, 90001])
@pytest.mark.parametrize("batches", [(1, 4), (4, 1)])
def test_plans_on_one_bank_give_the_same_bits(pkg, n, batches):
    """Statistics too (SIGMA), whatever the plans' sizes: the bank's plan decides the cut."""
    p = pkg.make_params(40, 2, 300, 20, stages=(1, 2), thresh=(6.0, 6.0), thresh_mode=pkg.THRESH_SIGMA, max_bins=n,
                        group_size=300, max_batch=batches[0])
    q = pkg.make_params(40, 2, 300, 20, stages=(1, 2), thresh=(6.0, 6.0), thresh_mode=pkg.THRESH_SIGMA,
                        max_bins=2 * n, max_batch=batches[1])
    x = torch.from_numpy(synth.spectrum(n, 97, [synth.Signal(n / 2.5, 20.0, 0.0, 30.0, 0.3)])).cuda()
    with pkg.Plan(p) as parent, parent.share(q) as child:
        got = []
        for plan in (parent, child):
            plan.search(x)
            found = [(c.stage, c.p, c.t, c.power) for c in plan.candidates()]
            got.append((found, plan.stats(0), [plan.maxproj(si)[0] for si in range(2)]))
        assert got[0][0] == got[1][0] and got[0][1] == got[1][1] and len(got[0][0]) > 0
        assert all(np.array_equal(a, b) for a, b in zip(got[0][2], got[1][2]))
        if max(batches) == child.params.max_batch:
            child.search_batch([x, x[: n // 2].contiguous()])
            child.candidates()
            assert child.stats(0) == got[0][1]
