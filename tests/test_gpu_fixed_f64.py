"""The FP64 step's integer arithmetic where its exponents can go wrong.

Dissipation, advection weights and T's transport are sums in 64-bit fixed point
scaled to the largest term, so: terms far apart (a field of 1e-25 beside one of
order 1, a single spike in zeros), fields that are zero or constant (exact zeros
have to stay zero), large weights (high Ra: advection above diffusion; low Ra:
below) and no dissipation at all (c4 = 0).  Against the FP64 oracle: a rate's
terms are of the size weight x field, ten steps round a few hundred times by
1.1e-16 of that, so 1e-12 of the max-norm.
"""
import numpy as np
import pytest

import oracle

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


def _state(kind, n):
    nx, ny, nz = n
    r = np.random.default_rng(5)
    q = np.zeros((5, nz, ny, nx))
    if kind == "rough":
        q[:] = r.uniform(-1.0, 1.0, q.shape)
    elif kind == "tiny_beside_large":
        q[:4] = 1e-25 * r.uniform(-1.0, 1.0, q[:4].shape)
        q[0, :, :, : nx // 2] *= 1e25
        q[4] = 0.5 * r.uniform(-1.0, 1.0, q[4].shape) * 10.0 ** r.integers(-30, 1, q[4].shape)
    elif kind == "spikes":
        for f in range(5):
            q[f, nz // 2, ny // 2 - 1, nx // 3 + f] = 0.7 - 0.3 * f
    elif kind == "constant":
        q[0], q[4] = 0.3, 0.25
    elif kind == "tiny":
        q[:] = 1e-270 * r.uniform(-1.0, 1.0, q.shape)
    return q


@pytest.mark.parametrize("kind", ["rough", "tiny_beside_large", "spikes", "constant", "tiny"])
@pytest.mark.parametrize("Ra,c4", [(1e7, 1.0 / 32.0), (10.0, 1.0 / 32.0), (1e5, 0.0)])
def test_fixed_point_rates_match_oracle(m, kind, Ra, c4):
    n = (35, 18, 21)
    q = _state(kind, n)
    o = oracle.OracleCavity(*n, dict(Ra=Ra, c4=c4))
    o.set_fields(q)
    o.step(10)
    with m.Cavity(*n, Ra=Ra, c4=c4) as c:
        c.set_fields(q)
        c.step(10)
        g, ref = c.fields(), o.fields()
        for f in range(5):
            assert np.max(np.abs(g[f] - ref[f])) <= 1e-12 * np.max(np.abs(ref[f])), f
        assert np.allclose(c.residual, o.residual, rtol=1e-11, atol=0)


@pytest.mark.parametrize("field", range(5))
@pytest.mark.parametrize("value", [np.nan, np.inf, -1e306])
def test_non_finite_values_stay_visible(m, field, value):
    """A NaN, an infinity or a value whose squares overflow at one node: the
    step reports a non-finite state, it does not turn it into numbers."""
    n = (35, 18, 21)
    q = _state("rough", n)
    q[field, 9, 8, 12] = value
    with m.Cavity(*n) as c:
        c.set_fields(q)
        try:
            c.step(2)
            bad = not np.all(np.isfinite(c.residual))
        except m.CavityError:
            bad = True
        assert bad
