"""jerk_plane for a range of templates: only the groups that hold one of them
are filtered, and the rows are the whole plane's, bit for bit, wherever the
range starts in its groups, at odd lengths and for output buffers on any
4-byte boundary."""
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


@pytest.mark.parametrize("n,seg_len,group_size,precision", [(9001, 0, 7, 0), (4096, 1024, 16, 0), (12345, 8192, 0, 0),
                                                            (1, 0, 5, 0), (9001, 0, 7, 2)])
def test_rows_of_a_range_are_the_whole_planes(pkg, n, seg_len, group_size, precision):
    p = pkg.make_params(12, 2, 40, 20, max_bins=n, seg_len=seg_len, group_size=group_size, precision=precision)
    x = torch.from_numpy(synth.spectrum(n, 41, [synth.Signal(n / 3, 4.0, 20.0, 30.0, 0.3)] if n > 64 else [])).cuda()
    with pkg.Plan(p) as plan:
        T = plan.info.n_templates
        whole = torch.empty(T, 2 * n, device="cuda")
        plan.plane(x, 0, T, whole)
        for t0, nt in ((0, 1), (T - 1, 1), (5, 9), (6, 14), (1, T - 2)):
            for shift in (0, 1, 2):                      # 16-, 4- and 8-byte starts
                buf = torch.full((nt * 2 * n + 8,), -1.0, device="cuda")
                plan.plane(x, t0, nt, buf[shift:])
                torch.cuda.synchronize()
                assert torch.equal(buf[shift:shift + nt * 2 * n].view(nt, 2 * n), whole[t0:t0 + nt])
                assert (buf[:shift] == -1).all() and (buf[shift + nt * 2 * n:] == -1).all()
