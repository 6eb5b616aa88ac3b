"""Relative error of off-grid powers at strong signals, against the direct sum in
64 bits.  Without acceleration the power sits in one or two bins, and the
roundings of a single bin's response show: a chain of 64 FP32 terms is off by
2.2e-7 (RMS), 16 terms and exact products by 0.8e-7; the limit, 1.2e-7, is what
summing every node at every bin reached (1.0e-7) and a fifth, for 96 points."""
import numpy as np
import pytest

import oracle
import synth
from parity import lib_ready

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("z,w", [(0.0, 0.0), (2.0, 0.0), (4.0, 0.0), (0.0, 20.0), (20.0, 60.0), (200.0, 600.0)])
def test_strong_signals(z, w):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg = lib_ready()
    n = 1 << 15
    rng = np.random.default_rng(int(10 * z + w))
    r = 1000.0 + 1000.0 * np.arange(24) + rng.uniform(0.0, 1.0, 24)
    F = (50.0 * synth.spectrum(n, 72, [synth.Signal(x, z, w, 40.0, float(rng.uniform(0, 6))) for x in r])).astype(
        np.complex64)
    points = [(x + d, z, w) for x in r for d in (0.0, 0.05, -0.1, 0.2)]
    p = pkg.make_params(4, 2, 20, 20, max_bins=n, norm_block=0)
    with pkg.Plan(p, build_templates=False) as plan:
        got = plan.power_at(torch.from_numpy(F).cuda(), points).astype(np.float64)
    want = np.array([oracle.power_at(F.astype(np.complex128), *q, pad=16) for q in points])
    rms = float(np.sqrt(np.mean(np.square(got / want - 1.0))))
    assert rms <= 1.2e-7, rms


def test_widest_windows():
    """The largest panel class (J = 1536, two node pairs at a time): windows of
    23 034 bins against the direct sum in 64 bits; 5e-7 is eight times the RMS error
    of wide windows (0.6e-7)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg = lib_ready()
    n, z, w = 1 << 15, 8000.0, 60000.0
    F = (50.0 * synth.spectrum(n, 73, [synth.Signal(16000.25, z, w, 400.0, 0.4)])).astype(np.complex64)
    points = [(16000.25, z, w), (16000.0, z, w), (14100.75, -z, w)]
    p = pkg.make_params(4, 2, 20, 20, max_bins=n, norm_block=0)
    with pkg.Plan(p, build_templates=False) as plan:
        got = plan.power_at(torch.from_numpy(F).cuda(), points).astype(np.float64)
    x, g = np.polynomial.legendre.leggauss(64)
    panels = 1300                                        # of 18 cycles at most
    u = torch.from_numpy((-0.5 + (np.arange(panels)[:, None] + 0.5 * (x + 1.0)) / panels).ravel()).cuda()
    g = torch.from_numpy(np.tile(g * 0.5 / panels, panels)).cuda()
    f = torch.from_numpy(F.astype(np.complex128)).cuda()
    want = []
    for r, pz, pw in points:
        mz = int(np.ceil(abs(pz) / 2.0 + abs(pw) / 8.0)) + 16
        k = torch.arange(max(0, int(np.ceil(r - mz))), min(n - 1, int(np.floor(r + mz))) + 1, device="cuda")
        phase = pz * u * u / 2.0 + pw * u ** 3 / 6.0
        node = torch.polar(g, 2.0 * np.pi * (phase - phase.round()))
        total = 0.0
        for part in k.split(512):
            turn = (part.double() - r)[:, None] * u[None, :]
            total = total + (f[part] * (torch.polar(torch.ones_like(turn), -2.0 * np.pi * (turn - turn.round()))
                                        @ node).conj()).sum()
        want.append(float(abs(total)) ** 2)
    assert np.max(np.abs(got / np.array(want) - 1.0)) <= 5e-7 * max(1.0, max(want) / min(want)) ** 0.5
    assert abs(got[0] / want[0] - 1.0) <= 5e-7
