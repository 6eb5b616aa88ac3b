"""Plan.search_subharmonic with room for many candidates: its record buffers hold
no more than the cells there are, so that four stages at once take less than the
two buffers of the asked-for size that one stage after another took; the results
are those of a call with little room, and too little room is an overflow."""
import numpy as np
import pytest

import synth
from parity import lib_ready

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_room_for_many_candidates():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg = lib_ready()
    n = 3000
    p = pkg.make_params(6, 2, 20, 20, stages=(1, 2, 3, 4), thresh=(3.0, 6.0, 8.0, 10.0), max_bins=n)
    x = torch.from_numpy(synth.spectrum(n, 64)).cuda()
    with pkg.Plan(p) as plan:
        few, stats, _ = plan.search_subharmonic(x, cap=2 * n)
        torch.cuda.synchronize()
        torch.cuda.reset_peak_memory_stats()
        before = torch.cuda.memory_allocated()
        cap = 1 << 24
        many, stats2, _ = plan.search_subharmonic(x, cap=cap)
        assert torch.cuda.max_memory_allocated() - before < 2 * cap * pkg.jerk.CANDIDATE_DTYPE.itemsize
        assert len(few) > 8 and many == few and np.array_equal(stats, stats2)
        with pytest.raises(pkg.JerkError) as e:
            plan.search_subharmonic(x, cap=1)
        assert e.value.code == pkg.jerk.JERK_EOVERFLOW
