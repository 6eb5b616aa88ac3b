"""jerk_subharmonic at the sizes where its tiling can go wrong (cells around a
block of 32, banks around the 1024-row index table, every H) and on planes
with zeros, infinities and values that are not numbers, against the same sums
formed by torch: FP32 in h order, the first maximum over ascending t, the
statistics of the FP32 sums in FP64."""
import ctypes

import pytest

from parity import lib_ready

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return lib_ready()


def near(a, h, H):
    q = (2 * abs(a) * h + H) // (2 * H)
    return q if a >= 0 else -q


@pytest.mark.parametrize("n,zmax,wmax,H,kind", [(1, 2, 20, 1, "plain"), (16, 6, 20, 2, "plain"), (17, 6, 0, 3, "plain"),
                                                (1000, 12, 40, 8, "plain"), (333, 62, 320, 4, "plain"),
                                                (250, 32, 320, 5, "plain"), (500, 6, 20, 6, "odd"),
                                                (500, 6, 20, 7, "large"), (500, 6, 20, 3, "tiny")])
def test_sums_equal_torch(pkg, n, zmax, wmax, H, kind):
    from paper_1911_01353_gb300 import jerk
    p = pkg.make_params(zmax, 2, wmax, 20, max_bins=max(n, 64), stages=(1,), thresh=(1.0,))
    g = torch.Generator(device="cuda").manual_seed(n + H)
    with pkg.Plan(p, build_templates=False) as plan:
        T, bN = plan.info.n_templates, 2 * n
        plane = torch.rand(T, bN, generator=g, device="cuda") * 8
        if kind == "odd":
            plane[:, 5] = float("nan")
            plane[3, 100] = float("nan")
            plane[4, 200] = float("inf")
            plane[:, 300:310] = 0.0
            plane[2, 400] = -3.0
        plane *= {"large": 1e25, "tiny": 1e-25}.get(kind, 1.0)
        M = torch.empty(bN, dtype=torch.int64, device="cuda")
        sums = torch.empty(2, dtype=torch.float64, device="cuda")
        st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        assert jerk.lib().jerk_subharmonic(plan._h, ctypes.c_void_p(plane.data_ptr()), n, H,
                                           ctypes.c_void_p(M.data_ptr()), ctypes.c_void_p(sums.data_ptr()), st) == 0
        torch.cuda.synchronize()
    nz, zc, wc = 2 * zmax // 2 + 1, zmax // 2, wmax // 20
    q = torch.arange(bN, device="cuda")
    best = torch.full((bN,), -1.0, device="cuda")
    arg = torch.zeros(bN, dtype=torch.int64, device="cuda")
    s1 = s2 = 0.0
    for t in range(T):
        zi, wi = t % nz - zc, t // nz - wc
        S = torch.zeros(bN, device="cuda")
        for h in range(1, H + 1):
            S = S + plane[(near(wi, h, H) + wc) * nz + near(zi, h, H) + zc][(2 * q * h + H) // (2 * H)]
        up = S > best
        best, arg = torch.where(up, S, best), torch.where(up, torch.full_like(arg, t), arg)
        s1, s2 = s1 + S.double().sum(), s2 + S.double().square().sum()
    got = M.view(torch.int32).view(-1, 2)
    assert torch.equal(got[:, 1].contiguous().view(torch.float32), best)
    assert torch.equal(~got[:, 0], arg.to(torch.int32))
    # pairs of FP32 keep about 2^-46 of a sum of up to 32 terms, FP64 the rest
    want = torch.stack((s1, s2))
    assert torch.allclose(sums, want, rtol=1e-12, atol=0.0, equal_nan=True)
