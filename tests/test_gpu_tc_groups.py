"""The tensor-core filter's two groups of warps: template groups of one, two and
odd numbers of templates, more than 256 templates per group (its 8-bit argmax),
one to three segments.  The stage-1 max-projection must be the maximum of the
plane rows of the same filter and the lowest template that reaches it, bit for
bit (both apply the same power scale to the same product)."""
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


@pytest.mark.parametrize("n,zmax,wmax,group_size,precision", [(1, 4, 0, 0, 2), (1500, 6, 20, 1, 2), (2500, 6, 20, 2, 1),
                                                              (5000, 6, 20, 7, 2), (5500, 40, 300, 2048, 2),
                                                              (5500, 40, 300, 513, 1), (9000, 60, 100, 0, 2)])
def test_max_projection_is_the_maximum_of_the_rows(pkg, n, zmax, wmax, group_size, precision):
    p = pkg.make_params(zmax, 2, wmax, 20, stages=(1,), thresh=(8.0,), thresh_mode=pkg.THRESH_SIGMA, max_bins=n,
                        group_size=group_size, precision=precision)
    sig = [synth.Signal(n / 2.5, zmax / 2.0, 0.0, 30.0, 0.3)] if n > 64 else []
    x = torch.from_numpy(synth.spectrum(n, 91, sig)).cuda()
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
        # the running maximum compares powers before their scale: equal scaled powers may differ there
        reaches = rows.cpu().numpy()[t, np.arange(bN)] == M
        assert reaches.all() and (t != first.cpu().numpy()).mean() < 1e-3
        d = rows.double()
        assert mu[0] == pytest.approx(float(d.mean()), rel=1e-6)
        assert sd[0] == pytest.approx(float(d.std(unbiased=False)), rel=1e-6)
