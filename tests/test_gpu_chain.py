"""Steps chained in graphs against the same steps one call at a time.

A call's steps run in graphs of 16, 4, 2 and 1 steps; inside a graph dt comes from
an atomic maximum, the centre shift from the state, and one finalise at the end
reduces every step's partials.  A call of one step finalises after it.  Fields,
dt, time and the records of the step log must not depend on the split: the
same sums in the same order, so equality is exact.
"""
import numpy as np
import pytest

import workloads

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


CASES = [
    ("fp64", (20, 17, 13), (1, 1, 1), False),
    ("fp64", (128, 128, 80), (1, 1, 1), False),  # stored walls between the steps
    ("fp64", (34, 30, 28), (2, 2, 2), False),
    ("fp64", (19, 22, 25), (1, 1, 1), True),
    ("fp32", (37, 21, 18), (1, 1, 1), False),
    ("fp32", (66, 34, 34), (2, 2, 2), False),
    ("fp32", (33, 17, 70), (1, 1, 1), True),
]


@pytest.mark.parametrize("prec,n,blocks,local", CASES)
def test_split_of_a_run_changes_nothing(m, prec, n, blocks, local):
    precision = m.CAVITY_FP64 if prec == "fp64" else m.CAVITY_FP32_MIXED
    kw = dict(blocks=blocks, precision=precision, seed=3, noise_amp=1e-3, Ra=3e4)
    q = workloads.smooth_state(n, seed=5)
    steps = 39  # 16 + 16 + 4 + 2 + 1
    got = []
    for calls in ([steps], [1] * steps, [3, 17, 5, 14]):
        with m.Cavity(*n, **kw) as c:
            log = m.cavity_step_log_alloc(16)  # shorter than the run: a ring
            m.cavity_set_step_log(c.h, log)
            if local:
                m.cavity_set_time_stepping(c.h, m.CAVITY_DT_LOCAL)
            c.step(2)
            c.set_fields(q)  # a refresh between graphs
            for k in calls:
                c.step(k)
            arrays = [m.cavity_get_block_array(c.h, b, f)[0] for b in range(m.cavity_num_blocks(c.h)) for f in (0, 4)]
            got.append((c.fields(), c.time, c.residual, c.nusselt, log.array.copy(), arrays))
            m.cavity_set_step_log(c.h, None)
            log.close()
    for other in got[1:]:
        assert np.array_equal(got[0][0], other[0])
        assert got[0][1] == other[1]
        assert np.array_equal(got[0][2], other[2])
        assert got[0][3] == other[3]
        for f in got[0][4].dtype.names:
            assert np.array_equal(got[0][4][f], other[4][f]), f
        for x, y in zip(got[0][5], other[5]):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_batch_split(m, prec):
    precision = m.CAVITY_FP64 if prec == "fp64" else m.CAVITY_FP32_MIXED
    sizes = [(24, 30, 27), (5, 4, 3), (40, 24, 33)]
    params = [m.cavity_default_params(Ra=r) for r in (1e3, 2e3, 3e4)]
    got = []
    for calls in ([21], [1] * 21):
        h = m.cavity_create_batch(sizes, params, precision=precision, noise_amp=1e-3)
        for k in calls:
            m.cavity_step(h, k)
        got.append([(m.cavity_batch_get_fields(h, b, n), m.cavity_batch_state(h, b)) for b, n in enumerate(sizes)])
        m.cavity_destroy(h)
    for (f0, s0), (f1, s1) in zip(*got):
        assert np.array_equal(f0, f1)
        assert (s0["step"], s0["t"], s0["dt"], s0["nusselt"]) == (s1["step"], s1["t"], s1["dt"], s1["nusselt"])
        assert np.array_equal(s0["residual"], s1["residual"])


def test_switching_the_overlapped_schedule_mid_run(m):
    kw = dict(blocks=(2, 1, 2), seed=3, noise_amp=1e-3, Ra=3e4)
    with m.Cavity(30, 22, 26, **kw) as a, m.Cavity(30, 22, 26, **kw) as b:
        a.step(25)
        b.step(6)
        m.cavity_set_overlap(b.h, True)
        b.step(9)
        m.cavity_set_overlap(b.h, False)
        b.step(10)
        assert np.array_equal(a.fields(), b.fields())
        assert a.time == b.time
