"""A cavity that just fits the GPU's memory.

The partials of sixteen steps are a percent of a large FP64 state.  Where they are what
no longer fits, the handle is created all the same and runs shorter graphs, with the
same results bit for bit.  (The memory is filled by one allocation that nothing touches.)
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MIB = 1 << 20


def _planes(m, c):
    nx, ny, nz = c.shape
    return m.cavity_get_fields_box(c.h, (1, 1, nz // 2), (nx, ny, 3))


@pytest.mark.parametrize("short", [24, 48])  # MiB less than the handle took: room for 4 sets, for 1
def test_handle_without_room_for_sixteen_sets(short):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2006_02602_gb300 as m
    n, kw = (384, 384, 384), dict(seed=3, noise_amp=1e-3, Ra=1e5)
    m.Cavity(8, 8, 8).close()  # the context and the kernels
    torch.cuda.empty_cache()
    free0 = torch.cuda.mem_get_info()[0]
    with m.Cavity(*n, **kw) as c:
        taken = free0 - torch.cuda.mem_get_info()[0]
        c.step(23)
        ref, t, res = _planes(m, c), c.time, c.residual
    free = torch.cuda.mem_get_info()[0]
    keep = taken - short * MIB
    filler = torch.empty((free - keep) // (2 * MIB) * (2 * MIB), dtype=torch.uint8, device="cuda")
    try:
        with m.Cavity(*n, **kw) as c:
            c.step(23)
            c.sync()
            del filler
            torch.cuda.empty_cache()
            assert np.array_equal(_planes(m, c), ref)
            assert c.time == t and np.array_equal(c.residual, res)
    finally:
        filler = None
        torch.cuda.empty_cache()
