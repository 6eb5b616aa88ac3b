"""jerk_power_at where its tiling can go wrong: windows shorter than one panel
class and as long as the call allows, points of several classes in one call,
points at and beyond the spectrum's ends, against the oracle's direct sum (FP32
arithmetic over windows of n bins: 1e-5 of the largest power)."""
import numpy as np
import pytest

import oracle
import synth
from parity import lib_ready

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return lib_ready()


@pytest.mark.parametrize("points", [
    [(100.3, 0.0, 0.0)],
    [(0.0, 0.0, 0.0), (-3.25, 4.0, 20.0), (3999.9, -8.0, 30.0), (4010.0, 2.0, 0.0), (9000.0, 0.0, 0.0)],
    [(2000.25, z, w) for z, w in ((0.5, 0.0), (33.3, -7.0), (-120.0, 60.0), (200.0, 600.0), (-700.0, 1500.0))],
    [(2000.75, 3000.0, -4000.0), (1500.5, 1.0, 1.0), (1999.0, -6000.0, 20000.0)],
])
def test_power_at_equals_the_direct_sum(pkg, points):
    n = 4000
    F = synth.spectrum(n, 71, [synth.Signal(2000.25, 33.0, -7.0, 40.0, 0.2)])
    p = pkg.make_params(4, 2, 20, 20, max_bins=n, norm_block=0)
    with pkg.Plan(p, build_templates=False) as plan:
        got = plan.power_at(torch.from_numpy(F).cuda(), points).astype(np.float64)
    want = np.array([oracle.power_at(F.astype(np.complex128), *q, pad=16) for q in points])
    assert np.max(np.abs(got - want)) <= 1e-5 * max(want.max(), 1.0)
