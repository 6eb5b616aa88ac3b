"""The harmonic sum's split of a spectrum's fundamentals over blocks (a spectrum
of few cells, many fundamentals) and its single launch over a batch: every
stage's max-projection is the maximum of the sums of plane rows, formed by torch
in FP32 in h order, with the lowest template on equal sums."""
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


@pytest.mark.parametrize("lengths,zmax,wmax,stages", [((900,), 20, 60, (1, 2)), ((5000,), 24, 120, (1, 2, 4, 8)),
                                                      ((2047, 1, 3000, 1025), 20, 100, (1, 3)),
                                                      ((40000,), 12, 40, (1, 2, 3, 4))])
def test_stage_maxima_are_the_row_sums(pkg, lengths, zmax, wmax, stages):
    total = sum(lengths)
    p = pkg.make_params(zmax, 2, wmax, 20, stages=stages, thresh=(1e9,) * len(stages), max_bins=total,
                        max_batch=len(lengths))
    xs = [torch.from_numpy(synth.spectrum(n, 81 + i)).cuda() for i, n in enumerate(lengths)]
    nz, nw = zmax + 1, wmax // 10 + 1
    with pkg.Plan(p) as plan:
        plan.search_batch(xs)
        plan.candidates()
        got = [[plan.maxproj_tensor(si, i).clone() for si in range(len(stages))] for i in range(len(xs))]
        for i, x in enumerate(xs):
            bN = 2 * x.numel()
            plane = torch.empty(nz * nw, bN, device="cuda")
            plan.plane(x, 0, nz * nw, plane)
            torch.cuda.synchronize()
            for si, H in enumerate(stages):
                n = (bN - 1) // H + 1
                best = torch.zeros(n, device="cuda")
                arg = torch.full((n,), -1, dtype=torch.int64, device="cuda")
                for t in range(nz * nw):
                    z, w = -zmax + 2 * (t % nz), -wmax + 20 * (t // nz)
                    if H * abs(z) > zmax or H * abs(w) > wmax:
                        continue
                    S = torch.zeros(n, device="cuda")
                    for h in range(1, H + 1):
                        th = (h * w + wmax) // 20 * nz + (h * z + zmax) // 2
                        S = S + plane[th][::h][:n]
                    up = (S > best) | (arg < 0)
                    best, arg = torch.where(up, S, best), torch.where(up, torch.full_like(arg, t), arg)
                u = got[i][si].view(torch.int32).view(-1, 2)
                assert torch.equal(u[:, 1].contiguous().view(torch.float32), best), (i, H)
                assert torch.equal(~u[:, 0], arg.to(torch.int32)), (i, H)
