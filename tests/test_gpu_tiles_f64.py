"""The FP64 step's tiles of consecutive nodes, at the sizes where they can go wrong.

A tile is 128 (BDC_F64_TY=8: 256) consecutive nodes of a plane over a chunk of
planes; the chunk depths depend on the size (4-plane and 1-plane tiles, or
8-plane and 2-plane ones from 64 tile planes an SM on).  The sizes below put
the last tile of a plane at one node, at a full tile and in between, a tile
over many rows (nx = 2, 3), and a plane count that leaves a remainder of both
chunk depths.  Fields against the FP64 oracle within 1e-12 of the max-norm:
a few hundred roundings of 1.1e-16 in ten steps.
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


def _check(m, n, steps, blocks=(1, 1, 1), Ra=1e5):
    o = oracle.OracleCavity(*n, dict(Ra=Ra), noise=1e-3, seed=2)
    o.step(steps)
    with m.Cavity(*n, blocks=blocks, seed=2, noise_amp=1e-3, Ra=Ra) as c:
        c.step(steps)
        g, ref = c.fields(), o.fields()
        for f in range(5):
            assert np.max(np.abs(g[f] - ref[f])) <= 1e-12 * np.max(np.abs(ref[f])), (n, blocks, f)
        assert np.allclose(c.residual, o.residual, rtol=1e-11, atol=0)
        assert np.allclose(c.nusselt, o.nusselt, rtol=1e-12, atol=0)
        assert c.time[1] == pytest.approx(o.t, rel=1e-13)


@pytest.mark.parametrize("n,blocks", [
    ((43, 3, 7), (1, 1, 1)),     # a plane of 129 nodes: the last tile holds one
    ((32, 4, 9), (1, 1, 1)),     # exactly one tile a plane
    ((2, 130, 5), (1, 1, 1)),    # 64 rows a tile
    ((127, 2, 6), (1, 1, 1)),
    ((67, 61, 71), (1, 1, 1)),   # 4-plane tiles below fine ones
    ((97, 33, 91), (4, 2, 1)),   # the same in ragged blocks
    ((101, 99, 140), (1, 1, 1)),  # 8-plane tiles below 2-plane ones, odd remainders
])
def test_tiles_match_oracle(m, n, blocks):
    _check(m, n, 10, blocks, Ra=3e4)


def test_256_node_tiles_match_oracle(m, monkeypatch):
    monkeypatch.setenv("BDC_F64_TY", "8")
    _check(m, (51, 37, 45), 10)


def test_sqrt_at_the_ends_of_its_binades(m):
    """m next to 1, 2 and 4 (the clamps of the FP32 pair) and next to perfect squares, all exponents' parities."""
    k = np.arange(-40, 41, dtype=np.int64)
    near = np.concatenate([(np.array([b]).view(np.int64) + k).view(np.float64)
                           for b in (0.25, 0.5, 1.0, 2.0, 4.0, 2.25, 1e300, 3.0e-38)])
    wide = np.concatenate([4.0 - 2.0 ** np.arange(-51, 0), 1.0 + 2.0 ** np.arange(-52, 0)])
    sq = np.random.default_rng(3).uniform(1.0, 2.0, 1 << 16) ** 2
    max_rel, n_diff = m.cavity_check_sqrt(np.concatenate([near, wide, sq]))
    assert max_rel <= 2.0 ** -52
