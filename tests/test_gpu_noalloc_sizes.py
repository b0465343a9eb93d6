"""The allocation-free step over the sizes where its tiling changes.

Tiles are 128 consecutive nodes of a plane, 1, 2, 4 or 8 planes deep by size,
deeper where the fixed scratch has no room, and 256 nodes where even 16 planes
of 128 do not fit.  Each size against cavity_step from the same state: the same
kernel arithmetic, so 1e-13 of the max-norm, and the norms' sums in another
order, 1e-12.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(17, 9, 5), (2, 3, 2), (64, 61, 45), (64, 64, 81), (130, 129, 101), (600, 300, 91),
                               (1536, 2048, 3)])
def test_noalloc_matches_cavity_step(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2006_02602_gb300 as m
    with m.Cavity(*n, seed=3, noise_amp=1e-3, Ra=2e4) as c:
        small = n[0] * n[1] * n[2] < 1 << 22
        if small:
            c.set_fields(workloads.smooth_state(n, seed=8))
        q_in = torch.stack([torch.from_numpy(m.cavity_get_block_array(c.h, 0, f)[0]) for f in range(5)]).cuda()
        q_out = torch.zeros_like(q_in)
        out6 = torch.zeros(6, dtype=torch.float64, device="cuda")
        _, _, dt = c.time
        for _ in range(2):  # twice: the scratch of the first call does not reach the second
            m.cavity_step_block_noalloc(q_in.data_ptr(), q_out.data_ptr(), n, c.params, dt, 0.0, out6.data_ptr(),
                                        torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        c.step(1)
        inner = (slice(2, -2),) * 3
        for f in range(5):
            ref = m.cavity_get_block_array(c.h, 0, f)[0][inner]
            got = q_out[f].cpu().numpy()[inner]
            assert np.max(np.abs(got - ref)) <= 1e-13 * max(np.max(np.abs(ref)), 1e-300), f
        res = out6.cpu().numpy()
        assert np.allclose(res[:5], c.residual, rtol=1e-12, atol=0)
        assert res[5] == pytest.approx(c.time[2], rel=1e-13)
