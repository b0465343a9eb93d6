"""The step log during the adjoint's reverse sweep.

The sweep recomputes every segment's steps but its last, and their records are written
again: into a log attached after the forward run come exactly those, equal to the
forward run's bit for bit.  The gradient is that of a sweep without a log.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n", [("fp64", (20, 14, 11)), ("fp64", (128, 128, 80)), ("fp32", (37, 14, 21))])
def test_recomputed_steps_are_logged_again(prec, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2006_02602_gb300 as m
    steps, ckpt = 23, 6
    kw = dict(precision=m.CAVITY_FP64 if prec == "fp64" else m.CAVITY_FP32_MIXED, seed=3, noise_amp=1e-3, Ra=2e4)
    theta = workloads.wall_temperature(n[1], n[2], seed=5)
    first, again = m.StepLog(steps), m.StepLog(steps)
    with m.Cavity(*n, **kw) as c, m.Cavity(*n, **kw) as ref:
        for x in (c, ref):
            m.cavity_set_wall_temperature(x.h, 0, theta)
        m.cavity_set_step_log(c.h, first)
        assert m.cavity_adjoint_forward(c.h, steps, ckpt) == m.cavity_adjoint_forward(ref.h, steps, ckpt)
        m.cavity_set_step_log(c.h, again)
        g, gra = m.cavity_adjoint_backward(c.h, n[1], n[2])
        g0, gra0 = m.cavity_adjoint_backward(ref.h, n[1], n[2])
        m.cavity_set_step_log(c.h, None)
        assert np.array_equal(g, g0) and gra == gra0
        assert c.time == ref.time and np.array_equal(c.fields(), ref.fields())
    for k in range(1, steps + 1):
        if k % ckpt and k != steps:
            for f in first.array.dtype.names:
                assert np.array_equal(again.array[k - 1][f], first.array[k - 1][f]), (k, f)
        else:
            assert again.array[k - 1]["step"] == 0
    first.close()
    again.close()
