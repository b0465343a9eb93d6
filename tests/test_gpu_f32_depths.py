"""The FP32-mixed step's shallow z chunks, down to one plane.

Those are the depths small cavities take by size.  As every tile shape they change
only the order of the residual sums: fields and time equal a 32-plane chunk's bit for
bit, over plane counts with and without a remainder, undivided and in blocks.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,blocks", [((45, 38, 70), (1, 1, 1)), ((33, 9, 24), (1, 1, 1)), ((46, 20, 38), (2, 1, 2))])
def test_shallow_chunks_give_identical_fields(monkeypatch, n, blocks):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2006_02602_gb300 as m

    def run():
        with m.Cavity(*n, blocks=blocks, precision=m.CAVITY_FP32_MIXED, seed=4, noise_amp=1e-3, Ra=3e4) as c:
            c.step(21)
            return c.fields(), c.time, c.nusselt

    out = [run()]  # the depth that follows the size
    for depth in (32, 1, 2, 3, 4, 6, 8, 11, 12):
        monkeypatch.setenv("BDC_F32_TILE", f"8,{depth},4,3")
        out.append(run())
    for f, t, nu in out:
        assert np.array_equal(f, out[1][0])
        assert t == out[1][1]
        assert np.allclose(nu, out[1][2], rtol=1e-12, atol=0)
