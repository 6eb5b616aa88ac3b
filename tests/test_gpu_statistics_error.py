"""How far the statistics may be from the 64-bit sums of the same FP32 numbers.

Filters: an FP32 partial covers 16 cells x 32 templates.  One addition is off by
2.5e-8 (RMS, of the running sum), 32 of them by 8.2e-8 of the partial; a mean over
n partials by 8.2e-8 / sqrt(n).  With partials of twice the cells it would be
1.41 times that; the limit is 1.2 times, over 48 spectra (RMS good to a tenth).
The 16-bit filter's partials are the same.

Sub-harmonic sums: no further from the exact sum than FP64 additions in turn,
9e-16 (squares of FP32 numbers make them lean), which the test takes as 1e-15."""
import ctypes
import math

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


@pytest.mark.parametrize("precision", [0, 2])
def test_filter_partials(pkg, precision):
    # max_batch 2: the group is cut to about 100 templates, so most partials are full ones
    p = pkg.make_params(16, 2, 340, 20, stages=(1,), thresh=(8.0,), thresh_mode=pkg.THRESH_SIGMA, max_bins=20000,
                        max_batch=2, group_size=1024, precision=precision)
    off = []
    with pkg.Plan(p) as plan:
        T = plan.info.n_templates
        for seed in range(48):
            n = 7000 + 61 * seed
            x = torch.from_numpy(synth.spectrum(n, 500 + seed)).cuda()
            rows = torch.empty(T, 2 * n, device="cuda")
            plan.plane(x, 0, T, rows)
            plan.search(x)
            mu, _, _ = plan.stats()
            off.append((mu[0] / float(rows.double().mean()) - 1.0) * math.sqrt(2.0 * n * T / (16 * 32)))
    rms = float(np.sqrt(np.mean(np.square(off))))
    assert rms <= 1.2 * 8.2e-8, rms


@pytest.mark.parametrize("H", [1, 2, 4, 8])
def test_subharmonic_sums(pkg, H):
    n, zmax, wmax = 16000, 20, 60
    nz, zc, wc = zmax + 1, zmax // 2, wmax // 20
    T, bN = nz * (2 * wc + 1), 2 * n
    p = pkg.make_params(zmax, 2, wmax, 20, stages=(1,), thresh=(1e9,), max_bins=n)
    off = []
    with pkg.Plan(p) as plan:
        for seed in range(8):
            x = torch.from_numpy(synth.spectrum(n, 600 + seed)).cuda()
            rows = torch.empty(T, bN, device="cuda")
            plan.plane(x, 0, T, rows)
            M = torch.empty(bN, dtype=torch.int64, device="cuda")
            sums = torch.empty(2, dtype=torch.float64, device="cuda")
            code = pkg.jerk.lib().jerk_subharmonic(plan._h, ctypes.c_void_p(rows.data_ptr()), n, H,
                                                   ctypes.c_void_p(M.data_ptr()), ctypes.c_void_p(sums.data_ptr()),
                                                   ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
            assert code == 0
            q = torch.arange(bN, device="cuda")

            def near(a, h):
                r = (2 * abs(a) * h + H) // (2 * H)
                return r if a >= 0 else -r
            S = torch.zeros(T, bN, device="cuda")
            for h in range(1, H + 1):
                t = [(near(i // nz - wc, h) + wc) * nz + near(i % nz - zc, h) + zc for i in range(T)]
                S += rows[torch.as_tensor(t, device="cuda")][:, (2 * q * h + H) // (2 * H)]
            S = S.cpu().numpy().astype(np.float64).ravel()
            got = sums.cpu().numpy()
            off.append((got[0] / math.fsum(S) - 1.0, got[1] / math.fsum(S * S) - 1.0))   # S^2 is exact
    rms = np.sqrt(np.mean(np.square(off), axis=0))
    assert (rms <= 1.0e-15).all(), rms
