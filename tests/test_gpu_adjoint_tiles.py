"""The adjoint sweep where its tiles meet.

A CTA sweeps 32 x 8 columns over a chunk of planes and takes its neighbours'
coefficients from a halo: several tiles along x and y with ragged last ones, one node
beyond a tile, exactly full ones.  Against the oracle's discrete adjoint, elementwise,
with the bounds of the single-tile sizes: FP64 1e-9 and FP32-mixed 1e-4 of the largest
component, Ra within the same.
"""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [(45, 19, 14), (33, 9, 23), (64, 16, 10), (71, 17, 5)])
def test_sweep_matches_oracle_across_tiles(n, prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2006_02602_gb300 as m
    Ra, steps = 2e4, 13
    theta = workloads.wall_temperature(n[1], n[2], seed=5)
    jo, go, grao = oracle.nusselt_gradient(*n, dict(Ra=Ra, Pr=0.71), steps, seed=3, noise=1e-3, t_hot_wall=theta)
    fp64 = prec == "fp64"
    with m.Cavity(*n, precision=m.CAVITY_FP64 if fp64 else m.CAVITY_FP32_MIXED, seed=3, noise_amp=1e-3, Ra=Ra,
                  Pr=0.71) as c:
        m.cavity_set_wall_temperature(c.h, 0, theta)
        j = m.cavity_adjoint_forward(c.h, steps, 5)
        g, gra = m.cavity_adjoint_backward(c.h, n[1], n[2])
    tol = 1e-9 if fp64 else 1e-4
    assert j == pytest.approx(jo, rel=1e-12 if fp64 else 1e-5)
    assert np.max(np.abs(g - go)) <= tol * np.max(np.abs(go))
    assert gra == pytest.approx(grao, rel=tol)
