"""A wall temperature set between the adjoint's forward run and its reverse sweep.

cavity_adjoint_backward returns the gradient of the last forward run's J.  The sweep
recomputes that run's states, so it has to do so with that run's wall temperature,
whatever the handle has been given since (the next iterate of an optimisation, say):
the same gradient bit for bit as without.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_gradient_is_of_the_forward_runs_walls(prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2006_02602_gb300 as m
    n, steps, ckpt = (20, 14, 11), 23, 6
    theta = workloads.wall_temperature(n[1], n[2], seed=5)
    got = []
    for between in (False, True):
        with m.Cavity(*n, precision=m.CAVITY_FP64 if prec == "fp64" else m.CAVITY_FP32_MIXED, seed=3,
                      noise_amp=1e-3, Ra=2e4) as c:
            m.cavity_set_wall_temperature(c.h, 0, theta)
            j = m.cavity_adjoint_forward(c.h, steps, ckpt)
            if between:
                m.cavity_set_wall_temperature(c.h, 0, 1.3 * theta)
            got.append((j, *m.cavity_adjoint_backward(c.h, n[1], n[2])))
    assert got[0][0] == got[1][0]
    assert np.array_equal(got[0][1], got[1][1])
    assert got[0][2] == got[1][2]
