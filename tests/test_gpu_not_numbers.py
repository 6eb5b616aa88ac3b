"""Bins that are not numbers, in every filter (the FP32 ones at each segment
length, the 16-bit ones): a segment that holds such a bin has no powers, but the
template groups' segments start at different cells, and where some template has
a power the max-projection is the largest of them, by the template that has it;
where none has, it is 0.  Powers are the plane rows of the same plan."""
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


@pytest.mark.parametrize("seg_len,precision", [(1024, 0), (2048, 0), (8192, 0), (4096, 0), (0, 1), (0, 2)])
@pytest.mark.parametrize("value", [complex(np.nan, 1.0), complex(1.0, np.inf)])
def test_maxima_are_those_of_the_numbers(pkg, seg_len, precision, value):
    n = 40000
    F = synth.spectrum(n, 63)
    F[[40, 5000, n - 1]] = np.complex64(value)
    p = pkg.make_params(40, 2, 160, 20, stages=(1,), thresh=(1e9,), seg_len=seg_len, precision=precision, max_bins=n,
                        norm_block=0, group_size=64)
    x = torch.from_numpy(F).cuda()
    with pkg.Plan(p) as plan:
        rows = torch.empty(plan.info.n_templates, 2 * n, device="cuda")
        plan.plane(x, 0, rows.shape[0], rows)
        plan.search(x)
        plan.candidates()
        M, t = plan.maxproj(0)
    power = torch.where(torch.isnan(rows), torch.full_like(rows, -1.0), rows)
    best = power.max(dim=0).values.cpu().numpy()
    some = torch.isnan(rows).any(dim=0).cpu().numpy()
    none = best < 0
    assert none.any() and (some & ~none).any() and not some.all()
    assert np.array_equal(M, np.where(none, np.float32(0), best))
    cell = np.flatnonzero(~none)
    assert np.array_equal(power.cpu().numpy()[t[cell], cell], best[cell])
    assert (t[none] == 0xFFFFFFFF).all()
