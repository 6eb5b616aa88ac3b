"""The L = 4096 filter's own edges: one to four segments (three share a CTA),
ragged ends, half-widths that drop no, one or two outputs per thread, template
groups shorter and longer than the 256 templates of its 8-bit argmax.  The
stage-1 max-projection must be the maximum of the plane rows it computes and
the lowest template that reaches it, the statistics those rows' sums (FP32
partials over 32 templates: 1e-6 relative), and a spectrum that is not a number
somewhere must leave the cells its filters do not reach unchanged."""
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


@pytest.mark.parametrize("n,zmax,wmax,group_size", [(1, 4, 0, 0), (1979, 6, 20, 7), (1981, 6, 20, 3), (3970, 6, 20, 0),
                                                    (6001, 40, 300, 300), (6001, 40, 300, 256), (20011, 60, 400, 0),
                                                    (9000, 200, 600, 2048)])
def test_max_projection_is_the_maximum_of_the_rows(pkg, n, zmax, wmax, group_size):
    p = pkg.make_params(zmax, 2, wmax, 20, stages=(1,), thresh=(8.0,), thresh_mode=pkg.THRESH_SIGMA, seg_len=4096,
                        max_bins=n, group_size=group_size)
    sig = [synth.Signal(n / 2.5, zmax / 2.0, 0.0, 30.0, 0.3)] if n > 64 else []
    x = torch.from_numpy(synth.spectrum(n, 61, sig)).cuda()
    with pkg.Plan(p) as plan:
        T, bN = plan.info.n_templates, 2 * n
        plan.search(x)
        plan.candidates()
        M, t = plan.maxproj(0)
        mu, sd, _ = plan.stats()
        rows = torch.empty(T, bN, device="cuda")
        plan.plane(x, 0, T, rows)
        torch.cuda.synchronize()
        best = rows.max(dim=0).values
        first = (rows == best).to(torch.uint8).argmax(dim=0)      # the lowest t
        assert np.array_equal(M, best.cpu().numpy())
        assert np.array_equal(t, first.cpu().numpy())
        d = rows.double()
        assert mu[0] == pytest.approx(float(d.mean()), rel=1e-6)
        assert sd[0] == pytest.approx(float(d.std(unbiased=False)), rel=1e-6)


def test_values_that_are_not_numbers_stay_where_the_filters_reach(pkg):
    n = 12000
    F = synth.spectrum(n, 62)
    bad = F.copy()
    bad[5000] = np.nan
    p = pkg.make_params(6, 2, 20, 20, stages=(1,), thresh=(1e9,), seg_len=4096, max_bins=n, norm_block=0)
    with pkg.Plan(p) as plan:
        got = []
        for f in (F, bad):
            plan.search(torch.from_numpy(f).cuda())
            plan.candidates()
            got.append(plan.maxproj(0))
        # cells of segments (at most 4096 cells long) that hold no such bin
        far = np.r_[0:2 * 5000 - 4096 - 64, 2 * 5000 + 4096 + 64:2 * n]
        assert np.array_equal(got[0][0][far], got[1][0][far]) and np.array_equal(got[0][1][far], got[1][1][far])
