"""The step log while a run goes on.

The device writes every step's record soon after the step, not once for many: a
host that reads the log during one long call sees, in a ring shorter than a graph of
16 steps, every step's record in its turn (a record stays for as many steps as the ring
holds, here twelve of half a millisecond or more, against a host loop of a few
microseconds).
"""
import time

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

CAP, STEPS = 12, 48


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


@pytest.mark.parametrize("prec,n,blocks", [
    ("fp64", (192, 192, 192), (1, 1, 1)),
    ("fp64", (190, 180, 170), (2, 2, 2)),
    ("fp32", (400, 320, 300), (1, 1, 1)),
    ("fp32", (400, 320, 300), (2, 2, 1)),
])
def test_every_step_is_seen_while_the_call_runs(m, prec, n, blocks):
    precision = m.CAVITY_FP64 if prec == "fp64" else m.CAVITY_FP32_MIXED
    log, after = m.StepLog(CAP), m.StepLog(STEPS)
    kw = dict(blocks=blocks, precision=precision, seed=2, noise_amp=1e-3, Ra=1e5)
    with m.Cavity(*n, **kw) as c, m.Cavity(*n, **kw) as ref:
        m.cavity_set_step_log(c.h, log)
        c.step(STEPS)
        seen = set()
        end = time.perf_counter() + 20.0
        while len(seen) < STEPS and time.perf_counter() < end and STEPS not in seen:
            for r in log.array:
                k = int(r["step"])
                if k:
                    seen.add(k)
        c.sync()
        seen.update(int(k) for k in log.array["step"])  # (the last two come together)
        assert sorted(seen) == list(range(1, STEPS + 1))
        m.cavity_set_step_log(ref.h, after)
        ref.step(STEPS)
        ref.sync()
        last = log.array[(STEPS - 1) % CAP]
        assert last["step"] == STEPS
        assert (last["t"], last["dt"]) == (ref.time[1], ref.time[2])
        m.cavity_set_step_log(c.h, None)
        m.cavity_set_step_log(ref.h, None)
        for k in range(max(1, STEPS - CAP + 1), STEPS + 1):
            assert np.array_equal(log.array[(k - 1) % CAP], after.array[k - 1])
    log.close()
    after.close()


def test_every_member_of_a_batch_is_seen(m):
    cavs = workloads.batch_cavities(ncav=32, nmin=64, nmax=96)
    h = m.cavity_create_batch([b["n"] for b in cavs], [m.cavity_default_params(Ra=1e4) for _ in cavs],
                              precision=m.CAVITY_FP64, noise_amp=1e-3)
    log = m.StepLog(CAP * len(cavs))
    try:
        m.cavity_set_step_log(h, log, CAP)
        m.cavity_step(h, STEPS)
        seen = [set() for _ in cavs]
        end = time.perf_counter() + 20.0
        while time.perf_counter() < end and any(STEPS not in s for s in seen):
            steps = log.array["step"].reshape(CAP, len(cavs)).copy()
            for q, s in enumerate(seen):
                s.update(int(k) for k in steps[:, q] if k)
        m.cavity_sync(h)
        steps = log.array["step"].reshape(CAP, len(cavs))
        for q, s in enumerate(seen):
            s.update(int(k) for k in steps[:, q])
            assert sorted(s) == list(range(1, STEPS + 1))
    finally:
        m.cavity_destroy(h)
        log.close()
