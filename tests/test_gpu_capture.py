"""Steps and stream captures.

A handle's steps run on its own stream, so they go on working while the same thread
captures another one, whatever they build on the way (a capture in global mode
forbids calls that allocate, and one made all the same ends it).  A capture of the
handle's own stream is refused, as a graph launch into one always is.
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


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_steps_while_another_stream_is_captured(m, prec):
    import torch
    precision = m.CAVITY_FP64 if prec == "fp64" else m.CAVITY_FP32_MIXED
    kw = dict(precision=precision, seed=3, noise_amp=1e-3, Ra=2e4)
    with m.Cavity(28, 25, 22, **kw) as c, m.Cavity(28, 25, 22, **kw) as ref:
        x = torch.ones(64, device="cuda")
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):  # (global capture mode)
            y = x * 2
            for _ in range(3):  # graphs are built meanwhile
                c.step(21)
        g.replay()
        torch.cuda.synchronize()
        assert float(y.sum()) == 128.0
        ref.step(63)
        assert np.array_equal(c.fields(), ref.fields())
        assert c.time == ref.time


@pytest.mark.filterwarnings("ignore:The CUDA Graph is empty")
def test_a_capture_of_the_handles_own_stream_is_refused_and_leaves_nothing_behind(m):
    import torch
    s = torch.cuda.Stream()
    with m.Cavity(20, 17, 15, seed=1, noise_amp=1e-3, stream=s.cuda_stream) as c:
        c.sync()
        g = torch.cuda.CUDAGraph()
        refused = False
        try:
            with torch.cuda.graph(g, stream=s):
                try:
                    c.step(3)
                except m.CavityError:
                    refused = True
        except RuntimeError:  # the refused launch may have ended the capture
            pass
        assert refused
        torch.cuda.synchronize()
        # the refusal is not the next call's error
        with m.Cavity(20, 17, 15, seed=1, noise_amp=1e-3) as a, m.Cavity(20, 17, 15, seed=1, noise_amp=1e-3) as b:
            a.step(5)
            for _ in range(5):
                b.step(1)
            assert np.array_equal(a.fields(), b.fields())
