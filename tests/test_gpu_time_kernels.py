"""Steps taken by cavity_time_kernels are steps of the run.

Under the overlapped schedule the shell nodes' kernel reads the stored walls, which
small FP64 cavities otherwise form where they are read: the event-timed steps
have to leave them stored as the schedule's own steps do.  The same arithmetic in
another order of launches, so equality is exact.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_02602_gb300 import build
    build.build()
    import paper_2006_02602_gb300 as mod
    mod.load_library()
    return mod


@pytest.mark.parametrize("n,blocks", [((30, 22, 26), (2, 1, 2)), ((41, 36, 29), (2, 2, 2))])
@pytest.mark.parametrize("timed", [1, 4])
def test_timed_steps_between_overlapped_ones(m, n, blocks, timed):
    kw = dict(blocks=blocks, seed=3, noise_amp=1e-3, Ra=3e4)
    with m.Cavity(*n, **kw) as a, m.Cavity(*n, **kw) as b:
        a.step(9 + timed)
        m.cavity_set_overlap(b.h, True)
        b.step(4)
        m.cavity_time_kernels(b.h, timed)
        b.step(5)
        assert np.array_equal(a.fields(), b.fields())
        assert a.time == b.time
