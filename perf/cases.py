"""What the speed of this framework is measured on: the calls its users make.

A case is a dict of plain values; its "kind" names the entry points it goes through:

run      one cavity (Cavity): advance `steps` steps, then read the fields, the residual norms, the Nusselt
         numbers and the time -- and, with "log", every step's record from the step log.  FP64 or FP32-mixed,
         undivided or split into blocks, global or local time stepping.
batch    a sweep of independent cavities of uneven sizes and Rayleigh numbers (cavity_create_batch, tuned once
         by cavity_autotune): advance all of them, then read every member's state and fields.
adjoint  the gradient of the mean hot-wall Nusselt number with respect to the hot-wall temperature field and Ra
         through autograd (mean_hot_wall_nusselt), as each iteration of an optimisation does.
block    one fused step of a block the caller holds in device memory (cavity_step_block_noalloc).

"start" is what a run begins from: "rest" (fluid at rest, conduction profile plus seeded noise) or "flow" (a
restart from a smooth seeded flow, set_fields).  A run goes on from where the last pass left it.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_2006_02602_gb300 as m
import workloads
from paper_2006_02602_gb300.autograd import mean_hot_wall_nusselt

PR, CFL, KAPPA, C4 = 0.71, 0.5, 0.1, 1.0 / 32.0  # the library's default parameters


# -- the cases ------------------------------------------------------------------

def _run(name, n, steps, fp32, ra, start, blocks=(1, 1, 1), noise=1e-3, local=False, log=False):
    return dict(name=name, kind="run", nx=n[0], ny=n[1], nz=n[2], px=blocks[0], py=blocks[1], pz=blocks[2],
                steps=steps, fp32=fp32, ra=float(ra), noise=noise, start=start, local=local, log=log)


def listed():
    return [
        # the small validation cavity, every step's residuals watched: launches and latency
        _run("fp64_32", (32, 32, 32), 200, False, 1e4, "rest", log=True),
        # a ragged cavity in pencils, restarted from a flow
        _run("fp64_97x65x50_4x2x1", (97, 65, 50), 100, False, 1e5, "flow", blocks=(4, 2, 1)),
        # the FP64 headline: 128^3 in eight blocks exchanging ghost faces
        _run("fp64_128_2x2x2", (128, 128, 128), 100, False, 1e5, "rest", blocks=(2, 2, 2)),
        # the largest single-GPU size timed in the paper, FP64
        _run("fp64_256", (256, 256, 256), 20, False, 1e5, "flow"),
        # a small ragged cavity in the FP32-mixed form: launches, latency, remainders of tiles
        _run("fp32_61x47x83", (61, 47, 83), 200, True, 1e4, "flow"),
        # the iteration in pseudo time towards a steady state: each node at its own step
        _run("fp32_96x80x72_local", (96, 80, 72), 200, True, 1e5, "rest", local=True),
        # the decomposed cavity in the FP32-mixed form
        _run("fp32_128_2x2x2", (128, 128, 128), 200, True, 1e5, "rest", blocks=(2, 2, 2)),
        # a large FP32-mixed run
        _run("fp32_256", (256, 256, 256), 200, True, 1e6, "flow", noise=1e-4),
        # the parameter sweep: 64 cavities of 24 .. 96 nodes an axis, Ra log-uniform from 1e3 up to 1e6 where the
        # size resolves it
        dict(name="batch64_fp32", kind="batch", ncav=64, nmin=24, nmax=96, steps=200, noise=1e-3),
        # one iteration of an optimisation over the hot wall's temperature
        dict(name="adjoint_fp32_128", kind="adjoint", nx=128, ny=128, nz=128, steps=200, ckpt=50, fp32=True, ra=1e5,
             noise=1e-3),
        # the same at the size gradients are validated at, in FP64
        dict(name="adjoint_fp64_32", kind="adjoint", nx=32, ny=32, nz=32, steps=40, ckpt=10, fp32=False, ra=1e5,
             noise=1e-3),
        # one step of a caller's block: a single call's latency
        dict(name="block_40x36x34", kind="block", nx=40, ny=36, nz=34, ra=1e5),
    ]


def _ra_cap(n):
    """The largest Ra a run on n nodes keeps going with: explicit Euler amplifies sound at the rate beta^2 dt / 2 of
    a diffusion, which the viscosity has to cover (0.3: a margin for both being shared by three axes)."""
    ra = 1e6
    while KAPPA * CFL * ra > 0.3 * (math.sqrt(KAPPA * ra * PR) * sum(a + 1 for a in n) + 2.0 * sum((a + 1) ** 2 for a in n)):
        ra *= 0.9
    return ra


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "run", "run", "batch", "adjoint", "adjoint", "block"])
    if kind == "batch":
        nmin = rng.randint(12, 40)
        return dict(kind="batch", ncav=_logint(rng, 8, 64), nmin=nmin, nmax=nmin + rng.randint(8, 56),
                    steps=rng.choice([50, 100, 200]), noise=1e-3)
    fp32 = rng.random() < 0.5
    pick_ra = lambda n: float(round(10.0 ** rng.uniform(3.0, math.log10(_ra_cap(n)))))  # noqa: E731
    if kind == "adjoint":
        n = [_logint(rng, 12, 112 if fp32 else 40) for _ in range(3)]
        return dict(kind="adjoint", nx=n[0], ny=n[1], nz=n[2], steps=rng.randint(20, 100 if fp32 else 40),
                    ckpt=rng.randint(7, 50), fp32=fp32, ra=pick_ra(n), noise=1e-3)
    if kind == "block":
        n = [_logint(rng, 16, 160) for _ in range(3)]
        return dict(kind="block", nx=n[0], ny=n[1], nz=n[2], ra=pick_ra(n))
    n = [_logint(rng, 16, 224) for _ in range(3)]
    blocks = rng.choice([(1, 1, 1), (1, 1, 1), (2, 2, 2), (4, 2, 1), (8, 1, 1)])
    if min(a // b for a, b in zip(n, blocks)) < 4:
        blocks = (1, 1, 1)
    # no dearer than the 256^3 runs
    most = (2.5e9 if fp32 else 2.5e8) / (n[0] * n[1] * n[2])
    steps = max(10, min(rng.choice([50, 100, 200, 301]), int(most)))
    local = rng.random() < 0.2
    c = _run("", n, steps, fp32, pick_ra(n), rng.choice(["rest", "flow"]), blocks=blocks, local=local, log=rng.random() < 0.3)
    del c["name"]
    return c


# -- inputs ---------------------------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _shape(c):
    return c["nx"], c["ny"], c["nz"]


def _flow(n, seed, ra):
    """A smooth seeded flow [5, nz, ny, nx] (p, u, v, w, T): low Fourier modes, no slip at the walls, speeds below
    the reference velocity sqrt(Ra Pr), T about the conduction profile; u, v, w in FP32 (both forms hold them)."""
    g = np.random.default_rng([seed, 7])
    dev = _device()
    z, y, x = torch.meshgrid(*[torch.arange(1, a + 1, dtype=torch.float64, device=dev) / (a + 1) for a in n[::-1]],
                             indexing="ij")
    uref = math.sqrt(ra * PR)
    out = torch.zeros(5, *z.shape, dtype=torch.float64, device=dev)
    for f, amp in enumerate((0.02 * uref * uref, 0.2 * uref, 0.2 * uref, 0.2 * uref, 0.1)):
        fn = torch.cos if f == 0 else torch.sin
        for _ in range(3):
            k = g.integers(1, 4, size=3) * math.pi
            out[f] += amp * g.uniform(-1, 1) * fn(k[0] * x) * fn(k[1] * y) * fn(k[2] * z)
    out[1:4] = out[1:4].float().double()
    out[4] += 1.0 - x
    return out


def _noise_state(n, seed, amp):
    """The library's initial state: at rest, T = 1 - x + amp (2U - 1), U from splitmix64(seed 2^40 + node)."""
    nx, ny, nz = n
    with np.errstate(over="ignore"):
        s = np.uint64(seed << 40) + np.arange(nx * ny * nz, dtype=np.uint64) + np.uint64(0x9E3779B97F4A7C15)
        s = (s ^ (s >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        s = (s ^ (s >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        s ^= s >> np.uint64(31)
    u = (s >> np.uint64(11)).astype(np.float64) / 9007199254740992.0
    q = np.zeros((5, nz, ny, nx))
    q[4] = 1.0 - np.arange(1, nx + 1) / (nx + 1) + amp * (2.0 * u.reshape(nz, ny, nx) - 1.0)
    return torch.from_numpy(q).to(_device())


def _seed(seed):
    return int(seed) % 1000003


def _start(c, seed):
    return _flow(_shape(c), _seed(seed), c["ra"]) if c["start"] == "flow" else \
        _noise_state(_shape(c), _seed(seed), c["noise"])


def _members(c, seed):
    r = np.random.default_rng([_seed(seed), 3])
    span = workloads.batch_cavities(c["ncav"], c["nmin"], c["nmax"])  # the sizes are the case's, not the seed's
    return [dict(n=b["n"], Ra=10.0 ** r.uniform(3.0, math.log10(_ra_cap(b["n"]))), seed=_seed(seed) + q) for q, b in enumerate(span)]


def _theta(c, seed):
    t = workloads.wall_temperature(c["ny"], c["nz"], seed=_seed(seed)).reshape(c["nz"], c["ny"])
    return torch.from_numpy(t).to(_device(), torch.float32 if c["fp32"] else torch.float64)


def _block_state(c, seed):
    one = torch.ones(c["nz"], c["ny"], dtype=torch.float64, device=_device())
    return _full(_flow(_shape(c), _seed(seed), c["ra"]), one, 0.0 * one)


def prepare(case, seed):
    c = case
    if c["kind"] == "run":
        s = m.Cavity(*_shape(c), blocks=(c["px"], c["py"], c["pz"]),
                     precision=m.CAVITY_FP32_MIXED if c["fp32"] else m.CAVITY_FP64, seed=_seed(seed),
                     noise_amp=c["noise"], Ra=c["ra"])
        if c["local"]:
            m.cavity_set_time_stepping(s.h, m.CAVITY_DT_LOCAL)
        if c["start"] == "flow":
            s.set_fields(_start(c, seed).cpu().numpy())
        log = None
        if c["log"]:
            log = m.cavity_step_log_alloc(c["steps"])
            m.cavity_set_step_log(s.h, log)
        # fields into page-locked memory, as a program that reads them again and again keeps it
        out = torch.empty(5, c["nz"], c["ny"], c["nx"], dtype=torch.float64, pin_memory=torch.cuda.is_available())
        return dict(c=c, cavity=s, log=log, out=out.numpy(), held=out)
    if c["kind"] == "batch":
        cavs = _members(c, seed)
        h = m.cavity_create_batch([b["n"] for b in cavs], [m.cavity_default_params(Ra=b["Ra"]) for b in cavs],
                                  seeds=[b["seed"] for b in cavs], noise_amp=c["noise"])
        m.cavity_autotune(h, 10)
        # every member's fields go one after another into one page-locked buffer, through the C entry point
        counts = [5 * b["n"][0] * b["n"][1] * b["n"][2] for b in cavs]
        out = torch.empty(sum(counts), dtype=torch.float64, pin_memory=torch.cuda.is_available())
        return _Batch(c, h, counts, out)
    if c["kind"] == "adjoint":
        ra = torch.tensor(c["ra"], dtype=torch.float32 if c["fp32"] else torch.float64)
        return dict(c=c, theta=_theta(c, seed).requires_grad_(), ra=ra.requires_grad_(), seed=_seed(seed))
    q = _block_state(c, seed)
    return dict(c=c, q=q, out=q.clone(), out6=torch.zeros(6, dtype=torch.float64, device=q.device),
                params=m.cavity_default_params(Ra=c["ra"]), dt=_block_dt(c))


class _Batch:
    """A batch handle, its members' value counts and the buffer for their fields; releases the handle."""

    def __init__(self, c, h, counts, out):
        self.c, self.h, self.counts, self.held, self.out = c, h, counts, out, out.numpy()
        self.at = [out.data_ptr() + 8 * sum(counts[:q]) for q in range(len(counts))]

    def __del__(self):
        m.cavity_destroy(self.h)


def _block_dt(c):
    # a stable step for speeds up to the reference velocity
    ih = [n + 1.0 for n in _shape(c)]
    return CFL / (2.0 * math.sqrt(c["ra"] * PR) * sum(ih) + 2.0 * sum(i * i for i in ih))


# -- one pass -------------------------------------------------------------------

def _residuals(res, fp32):
    # the FP32-mixed form's rates are FP32 numbers, and so are their norms
    return np.array(res, dtype=np.float32 if fp32 else np.float64)


def run(state):
    if isinstance(state, _Batch):
        h = state.h
        m.cavity_step(h, state.c["steps"])
        members = [m.cavity_batch_state(h, q) for q in range(len(state.counts))]
        get = m.load_library().cavity_batch_get_fields
        for q, (at, count) in enumerate(zip(state.at, state.counts)):
            if get(h, q, m.CAVITY_FIELD_ALL, ctypes.cast(at, ctypes.POINTER(ctypes.c_double)), count) != m.CAVITY_OK:
                raise RuntimeError(m.cavity_last_error(h))
        return dict(time=np.array([[b["t"], b["dt"]] for b in members]),
                    residual=_residuals([b["residual"] for b in members], True),
                    nusselt=np.array([b["nusselt"] for b in members]),
                    fields=state.out)
    c = state["c"]
    if c["kind"] == "run":
        s = state["cavity"]
        s.step(c["steps"])
        fields = s.fields(out=state["out"])
        _, t, dt = s.time
        got = dict(fields=fields, residual=_residuals(s.residual, c["fp32"]), nusselt=np.array(s.nusselt),
                   time=np.array([t, dt]))
        if state["log"] is not None:
            a = state["log"].array  # a ring as long as a pass: this pass's steps in their order
            got["log"] = dict(time=np.stack([a["t"], a["dt"]], 1), residual=_residuals(a["res"], c["fp32"]),
                              nusselt=np.stack([a["nu_hot"], a["nu_cold"]], 1))
        return got
    if c["kind"] == "adjoint":
        j = mean_hot_wall_nusselt(state["theta"], state["ra"], _shape(c), c["steps"], c["ckpt"],
                                  precision=m.CAVITY_FP32_MIXED if c["fp32"] else m.CAVITY_FP64, seed=state["seed"],
                                  noise=c["noise"])
        gtheta, gra = torch.autograd.grad(j, (state["theta"], state["ra"]))
        return dict(J=j.detach(), theta=gtheta, ra=gra)
    m.cavity_step_block_noalloc(state["q"].data_ptr(), state["out"].data_ptr(), _shape(c), state["params"],
                                state["dt"], 0.0, state["out6"].data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
    return dict(q=state["out"], norms=state["out6"])


# -- what a pass cannot do without ------------------------------------------------

# the five fields read once and written once a step (the FP32-mixed form holds p and T in two words), and the
# operations of the rates, the update, the norms and the stable step at one node
STEP_BYTES, STEP_FLOPS = {False: 80, True: 56}, 190


def work(case):
    c = case
    if c["kind"] == "batch":
        pts = sum(b["n"][0] * b["n"][1] * b["n"][2] for b in _members(c, 0))
        return dict(bytes=pts * (56 * c["steps"] + 40), flops=pts * STEP_FLOPS * c["steps"])
    pts = c["nx"] * c["ny"] * c["nz"]
    if c["kind"] == "block":
        return dict(bytes=80 * pts, flops=STEP_FLOPS * pts)
    if c["kind"] == "run":
        return dict(bytes=pts * (STEP_BYTES[c["fp32"]] * c["steps"] + 40), flops=pts * STEP_FLOPS * c["steps"])
    # forward, and backward the state and the adjoint read and the adjoint written, about twice the operations
    back = 28 + 40 if c["fp32"] else 40 + 80
    return dict(bytes=pts * (STEP_BYTES[c["fp32"]] + back) * c["steps"], flops=3 * pts * STEP_FLOPS * c["steps"])


# -- the same in 64 bits, written out plainly ---------------------------------------

def _ends(a, dim):
    n = a.shape[dim]
    return [a.narrow(dim, i, 1) for i in (0, 1, n - 1, n - 2)]


def _pad_p(p):
    for dim in (2, 1, 0):  # wall 2 p1 - p2 and the ghost beyond it 2 pw - p1
        a1, a2, b1, b2 = _ends(p, dim)
        p = torch.cat([3 * a1 - 2 * a2, 2 * a1 - a2, p, 2 * b1 - b2, 3 * b1 - 2 * b2], dim)
    return p


def _pad_t(t, hot, cold):
    t = torch.cat([hot[:, :, None], t, cold[:, :, None]], 2)  # isothermal x walls, the others adiabatic
    for dim in (1, 0):
        a1, a2, b1, b2 = _ends(t, dim)
        t = torch.cat([(4 * a1 - a2) / 3, t, (4 * b1 - b2) / 3], dim)
    return t


def _full(q, hot, cold):
    """The interior state with walls and ghosts, nodes -1 .. n+2 (edges and corners are read by no stencil)."""
    one = torch.nn.functional.pad(torch.cat([q[1:4], _pad_t(q[4], hot, cold)[None, 1:-1, 1:-1, 1:-1]]), (2,) * 6)
    one[3, 1:-1, 1:-1, 1:-1] = _pad_t(q[4], hot, cold)
    return torch.cat([_pad_p(q[0])[None], one])


def _at(a, wide, dim, off):
    """The interior window of an array padded by `wide`, moved by `off` along the last-but-`dim` axis."""
    ix = [slice(wide, s - wide) for s in a.shape[-3:]]
    s = ix[2 - dim]
    ix[2 - dim] = slice(s.start + off, s.stop + off)
    return a[(..., *ix)]


def _spectral(v, b2, ih):
    lam = 0.5 * (v.abs() + torch.sqrt(v * v + 4.0 * b2))
    return lam, sum(lam[d] * ih[d] for d in range(3)) + 2.0 * max(1.0, PR) * sum(i * i for i in ih)


def _b2(v, ra):
    floor = KAPPA * torch.clamp(torch.as_tensor(ra, dtype=torch.float64, device=v.device) * PR, min=1.0)
    return torch.maximum((v * v).sum(0), floor)


def _rates(q, p, vt, ra):
    """dq/dt of the interior and the stable-step bound of its nodes; p padded by 2, vt = u, v, w, T by 1."""
    n = q.shape[:0:-1]
    ih = [a + 1.0 for a in n]
    v = q[1:4]
    b2 = _b2(v, ra)
    lam, s = _spectral(v, b2, ih)
    r = 0.0
    div = diss = 0.0
    k = torch.tensor([PR, PR, PR, 1.0], dtype=torch.float64, device=q.device)[:, None, None, None]
    grad = []
    for d in range(3):
        up, dn = _at(vt, 1, d, 1), _at(vt, 1, d, -1)
        r = r - v[d] * (up - dn) * (0.5 * ih[d]) + k * (up - 2.0 * q[1:] + dn) * (ih[d] * ih[d])
        div = div + (up[d] - dn[d]) * (0.5 * ih[d])
        pp, pm = _at(p, 2, d, 1), _at(p, 2, d, -1)
        grad.append((pp - pm) * (0.5 * ih[d]))
        diss = diss + C4 * lam[d] * ih[d] * (_at(p, 2, d, 2) - 4.0 * pp + 6.0 * q[0] - 4.0 * pm + _at(p, 2, d, -2))
    zero = torch.zeros_like(div)
    buoy = ra * PR * (q[4] - 0.5)
    return torch.cat([(-b2 * div - diss)[None], r + torch.stack([-grad[0], -grad[1], buoy - grad[2], zero])]), s


def _centre_mean(p):
    ix = [slice((a - 1) // 2, a // 2 + 1) for a in p.shape]
    return p[tuple(ix)].mean()


def _step(q, hot, cold, ra, local):
    vt = torch.cat([torch.nn.functional.pad(q[1:4], (1,) * 6), _pad_t(q[4], hot, cold)[None]])
    r, s = _rates(q, _pad_p(q[0]), vt, ra)
    dt = CFL / s.reshape(-1)[s.reshape(-1).argmax()]
    new = q + (CFL / s if local else dt) * r
    return torch.cat([(new[0] - _centre_mean(new[0]))[None], new[1:]]), r, dt


def _nusselt(t, wall, high):
    ih = t.shape[2] + 1.0
    t1, t2 = (t[:, :, -1], t[:, :, -2]) if high else (t[:, :, 0], t[:, :, 1])
    flux = (3.0 * wall - 4.0 * t1 + t2).mean() * (0.5 * ih)
    return -flux if high else flux


def _advance(q, steps, ra, local, log=False):
    hot = torch.ones(q.shape[1:3], dtype=torch.float64, device=q.device)
    cold = torch.zeros_like(hot)
    ih = [a + 1.0 for a in q.shape[:0:-1]]
    next_dt = lambda q: CFL / _spectral(q[1:4], _b2(q[1:4], ra), ih)[1].max()  # noqa: E731
    nu = lambda q: torch.stack([_nusselt(q[4], hot, False), _nusselt(q[4], cold, True)])  # noqa: E731
    rms = lambda r: (r * r).mean((1, 2, 3)).sqrt()  # noqa: E731
    t, rows = torch.zeros((), dtype=torch.float64, device=q.device), []
    for _ in range(steps):
        q, r, dt = _step(q, hot, cold, ra, local)
        t = t + dt
        if log:
            rows.append((torch.stack([t, next_dt(q)]), rms(r), nu(q)))
    got = dict(fields=q, residual=rms(r), nusselt=nu(q), time=torch.stack([t, next_dt(q)]))
    if log:
        got["log"] = dict(zip(("time", "residual", "nusselt"), (torch.stack(x) for x in zip(*rows))))
    return got


def _adjoint(c, seed):
    theta = _theta(c, seed).double()
    cold = torch.zeros_like(theta)
    ra = torch.tensor(c["ra"], dtype=torch.float64, device=theta.device)
    q = _noise_state(_shape(c), _seed(seed), c["noise"])
    n, states = c["steps"], []
    for _ in range(n):
        states.append(q)
        q = _step(q, theta, cold, ra, False)[0]
    j, back = 0.0, torch.zeros_like(q)
    gtheta, gra = torch.zeros_like(theta), torch.zeros_like(ra)
    for q in reversed(states):
        with torch.enable_grad():
            x = [a.detach().requires_grad_() for a in (q, theta, ra)]
            new = _step(x[0], x[1], cold, x[2], False)[0]
            nu = _nusselt(new[4], x[1], False)
            back, a, b = torch.autograd.grad([new, nu], x, [back, torch.full_like(nu, 1.0 / n)])
        j, gtheta, gra = j + nu.detach() / n, gtheta + a, gra + b
    return dict(J=j, theta=gtheta, ra=gra)


def exact(case, seed):
    c = case
    with torch.no_grad():
        if c["kind"] == "run":
            return _advance(_start(c, seed), c["steps"], c["ra"], c["local"], c["log"])
        if c["kind"] == "batch":
            got = [_advance(_noise_state(b["n"], b["seed"], c["noise"]), c["steps"], b["Ra"], False)
                   for b in _members(c, seed)]
            keep = {k: torch.stack([g[k] for g in got]) for k in ("time", "residual", "nusselt")}
            return dict(keep, fields=torch.cat([g["fields"].reshape(-1) for g in got]))
        if c["kind"] == "adjoint":
            return _adjoint(c, seed)
        full, dt = _block_state(c, seed), _block_dt(c)
        q = full[:, 2:-2, 2:-2, 2:-2]
        r, _ = _rates(q, full[0], full[1:, 1:-1, 1:-1, 1:-1], c["ra"])
        out = full.clone()
        out[:, 2:-2, 2:-2, 2:-2] = q + dt * r
        v = out[1:4, 2:-2, 2:-2, 2:-2]
        s = _spectral(v, _b2(v, c["ra"]), [a + 1.0 for a in _shape(c)])[1]
        return dict(q=out, norms=torch.cat([(r * r).mean((1, 2, 3)).sqrt(), CFL / s.max().reshape(1)]))
