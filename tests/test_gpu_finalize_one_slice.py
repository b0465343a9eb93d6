"""The finalise of cavities whose partials fit one slice.

Then a step that is not a graph's last is finalised by one CTA: it folds the slice
and, FP64, the x walls' Nusselt partials through the same shared rows, which a barrier
keeps apart.  Without it a wall partial could be counted twice, now and then, in the
step log's Nusselt numbers and in the adjoint's J.  So many steps, every record of
which equals that of calls of one step (another path: the wall CTAs arrive at a
counter); the same sums in the same order, so equality is exact.
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


@pytest.mark.parametrize("n", [(16, 16, 16), (24, 24, 24), (20, 17, 13), (2, 3, 2)])
def test_every_record_equals_that_of_single_steps(m, n):
    steps = 320
    kw = dict(seed=3, noise_amp=1e-3, Ra=5e2)  # (stable at two nodes an axis)
    logs = [m.StepLog(steps) for _ in range(2)]
    with m.Cavity(*n, **kw) as a, m.Cavity(*n, **kw) as b:
        m.cavity_set_step_log(a.h, logs[0])
        m.cavity_set_step_log(b.h, logs[1])
        a.step(steps)
        for _ in range(steps):
            b.step(1)
        a.sync()
        b.sync()
        for f in logs[0].array.dtype.names:
            assert np.array_equal(logs[0].array[f], logs[1].array[f]), f
        nu = logs[1].array["nu_hot"].copy()
    with m.Cavity(*n, **kw) as c:
        j = m.cavity_adjoint_forward(c.h, steps, 16)
        acc = 0.0
        for v in nu:  # (the device's order)
            acc += v
        assert j == acc / steps
    for log in logs:
        log.close()
