"""The adjoint with a checkpoint segment longer than a grid's second dimension.

The argmax of a segment's states is taken by launches over (parts, states), of at
most 65535 states each; a segment may hold more (small cavities, long runs).  The
gradient does not depend on the checkpoint interval: 1e-12 of the largest component, as
between other intervals.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_segment_of_more_than_65535_states(prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2006_02602_gb300 as m
    n, steps = (2, 2, 2), 65600
    theta = workloads.wall_temperature(n[1], n[2], seed=6)
    got = []
    for ckpt in (steps, 4096):
        with m.Cavity(*n, precision=m.CAVITY_FP64 if prec == "fp64" else m.CAVITY_FP32_MIXED, seed=3,
                      noise_amp=1e-3, Ra=300.0) as c:
            m.cavity_set_wall_temperature(c.h, 0, theta)
            j = m.cavity_adjoint_forward(c.h, steps, ckpt)
            got.append((j, *m.cavity_adjoint_backward(c.h, n[1], n[2])))
    (j1, g1, r1), (j2, g2, r2) = got
    assert np.all(np.isfinite(g1)) and j1 == j2
    assert np.max(np.abs(g1 - g2)) <= 1e-12 * np.max(np.abs(g1))
    assert r1 == pytest.approx(r2, rel=1e-12)
