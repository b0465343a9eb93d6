"""The first call on a handle.

A call's steps run from graphs that are kept; the first time a piece of a call is
needed its kernels are launched as they are, so that no graph is built before the
GPU has work.  Results do not depend on which of the two a step came from
(test_gpu_chain's calls of every kind), and the first call's device time is that of its
steps.
"""
import numpy as np
import pytest

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


def test_first_call_takes_as_long_as_its_steps(m):
    import torch
    s = torch.cuda.Stream()
    extra = []
    for seed in range(7):
        with m.Cavity(160, 160, 160, precision=m.CAVITY_FP32_MIXED, seed=seed, noise_amp=1e-3, Ra=1e5,
                      stream=s.cuda_stream) as c:
            us = []
            for _ in range(6):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                c.sync()
                a.record(s)
                c.step(20)
                b.record(s)
                b.synchronize()
                us.append(1e3 * a.elapsed_time(b))
            extra.append(us[0] - min(us[2:]))
    # 20 steps of 66 us; building the graphs of 16 and 4 steps before the first launch takes 150 us and more
    assert np.median(extra) <= 80.0


def test_steps_repeat_bit_for_bit_from_launches_and_graphs(m):
    n = (30, 25, 22)
    for precision in (m.CAVITY_FP64, m.CAVITY_FP32_MIXED):
        for blocks in ((1, 1, 1), (2, 1, 2)):
            kw = dict(blocks=blocks, precision=precision, seed=3, noise_amp=1e-3, Ra=2e4)
            with m.Cavity(*n, **kw) as a, m.Cavity(*n, **kw) as b:
                for k in (23, 23, 23, 1, 1, 1, 23):  # launched, then from graphs, at both parities
                    a.step(k)
                for _ in range(3 * 23 + 3 + 23):
                    b.step(1)
                assert np.array_equal(a.fields(), b.fields())
                assert a.time == b.time and a.nusselt == b.nusselt
                assert np.array_equal(a.residual, b.residual)
