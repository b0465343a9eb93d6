"""A wall temperature set between the adjoint's forward run and its reverse sweep.

cavity_adjoint_backward returns the gradient of the last forward run's J.  The sweep
recomputes that run's states, so it has to do so with that run's wall temperature,
whatever the handle has been given since (the next iterate of an optimisation, say):
the same gradient bit for bit as without.  The state it leaves is the one after the
forward run, from which the handle goes on with what it has been given since.
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


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("setter", ["wall", "params"])
def test_the_run_goes_on_with_what_was_set_between(prec, setter):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2006_02602_gb300 as m
    n, steps = (20, 14, 11), 23
    theta = workloads.wall_temperature(n[1], n[2], seed=5)
    kw = dict(precision=m.CAVITY_FP64 if prec == "fp64" else m.CAVITY_FP32_MIXED, seed=3, noise_amp=1e-3, Ra=2e4)

    def change(c):
        if setter == "wall":
            m.cavity_set_wall_temperature(c.h, 0, 1.3 * theta)
        else:
            m.cavity_set_params(c.h, m.cavity_default_params(Ra=5e3))

    with m.Cavity(*n, **kw) as a, m.Cavity(*n, **kw) as b:
        for c in (a, b):
            m.cavity_set_wall_temperature(c.h, 0, theta)
        m.cavity_adjoint_forward(a.h, steps, 6)
        change(a)
        m.cavity_adjoint_backward(a.h, n[1], n[2])
        b.step(steps)
        change(b)
        assert a.time == b.time
        for _ in range(5):  # both buffer sets
            a.step(1)
            b.step(1)
        assert np.array_equal(a.fields(), b.fields())
        assert a.time == b.time and a.nusselt == b.nusselt
