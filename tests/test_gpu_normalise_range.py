"""The normaliser bit for bit against NumPy in FP64 where a block's scale factor
is small enough that its FP32 remainder, or the factor itself, is subnormal
(moduli of 1e31 and above), and at the largest factors."""
import numpy as np
import pytest

from parity import lib_ready
from test_gpu_normalise_edges import want

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("B", [100, 1024, 4096])
@pytest.mark.parametrize("amplitude", [1e-37, 1e-33, 1e-29, 1e29, 1e31, 1e33, 1e34, 1e35, 1e36, 5e37])
def test_scale_of_any_size(amplitude, B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg = lib_ready()
    n = 1 << 18
    rng = np.random.default_rng(int(np.log10(amplitude)) + 100 * B)
    F = (np.clip(rng.standard_normal(n), -4, 4) + 1j * np.clip(rng.standard_normal(n), -4, 4)).astype(np.complex64)
    F *= np.float32(amplitude)
    assert np.isfinite(F.real).all() and np.isfinite(F.imag).all()
    p = pkg.make_params(2, 2, 0, 20, max_bins=64, norm_block=B)
    ref = want(F, B)
    with pkg.Plan(p, build_templates=False) as plan:
        x = torch.from_numpy(F).cuda()
        y = torch.empty_like(x)
        plan.normalise(x, y)
        torch.cuda.synchronize()
    got = y.cpu().numpy()
    assert np.array_equal(got.real, ref.real) and np.array_equal(got.imag, ref.imag)
