"""The workloads whose speed is measured: what a program does with this framework, through
its public entry points (the package's ``Engine``, ``Server``, ``Hydro`` and ``Surrogate``).

Sizes and state points are those of the repository's own workloads (``workloads.py``,
``bench.py``, the README's example and the tests): 108-4000-atom EOS batches, one 4000-atom
query, boxes up to 32000 atoms, the 256-32000-atom serving mix, the 2000-zone coupled shock
tube, and the 4-member surrogate ensemble.

Every answer comes back whole and in its own type.  An MD answer of a few hundred steps or
more is a point of a chaotic trajectory: it has no 64-bit value to compare with (a rounding
in the first step changes every digit of it), so ``exact`` gives one for short runs only,
and for the parts that are not trajectories (hydro with an analytic closure, the networks).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2508_06012_gb300 as m
from paper_2508_06012_gb300 import workloads as W

RHO_UNEVEN, T_UNEVEN = (0.3, 1.2), (0.7, 3.0)    # the uneven batch and the serving stream
RHO_SMALL, T_SMALL = (0.5, 1.0), (1.0, 2.0)      # the 16 x 256-atom queries
NORM = (0.75, -1.0, 0.25, 2.0, 1.5, 1.2, 2.0, 0.6)  # normalisers of the inference benchmark
NPARAM, H = 33666, 128


def listed():
    return [
        # the smallest call: one element asks once, few steps; latency of the whole call
        dict(name="query_256_short", kind="query", nbox=1, sizes="fixed", natoms=256, lo=0, hi=0,
             steps_equil=50, steps_avg=50),
        # 16 independent 256-atom queries at once, 1000 + 1000 steps
        dict(name="queries_16x256", kind="query", nbox=16, sizes="fixed", natoms=256, lo=0, hi=0,
             steps_equil=1000, steps_avg=1000),
        # one 4000-atom query, 1000 + 1000 steps (the README's example; the paper's box)
        dict(name="query_4000", kind="query", nbox=1, sizes="fixed", natoms=4000, lo=0, hi=0,
             steps_equil=1000, steps_avg=1000),
        # the benchmark's uneven batch (N = 4 n^3, n = 3..10), a quarter of its boxes
        dict(name="batch_uneven_1024", kind="query", nbox=1024, sizes="fcc", natoms=0, lo=3, hi=10,
             steps_equil=1000, steps_avg=1000),
        # ragged atom counts, every force path (two boxes per SM)
        dict(name="batch_ragged_304", kind="query", nbox=304, sizes="log", natoms=0, lo=40, hi=4096,
             steps_equil=200, steps_avg=200),
        # one box of the largest size in use, state in device memory
        dict(name="query_32000", kind="query", nbox=1, sizes="fixed", natoms=32000, lo=0, hi=0,
             steps_equil=200, steps_avg=200),
        # the serving mix in a closed loop: queue, persistent grid, results by polling
        dict(name="serve_mix_304", kind="serve", nreq=304, lo=256, hi=32000, steps_equil=100,
             steps_avg=100),
        # one coupled hydro step: every zone's 500-atom box from its stored state
        dict(name="coupled_2000x500", kind="coupled", zones=2000, natoms=500, steps_equil=200,
             steps_avg=300, first_equil=600, first_avg=300),
        # the hydro caller with an analytic closure
        dict(name="hydro_ideal_2000", kind="hydro", zones=2000, closure="ideal", steps=200),
        # surrogate ensemble, device-resident queries
        dict(name="infer_1m", kind="infer", n=1 << 20, chunk=1 << 18),
        # surrogate ensemble asked from host arrays: one hydro step's worth of zones
        dict(name="predict_2000", kind="predict", n=2000, chunk=4096),
        # one epoch of the surrogate's training
        dict(name="train_32k", kind="train", n=32768, batch=512, epochs=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "one", "uneven", "ragged", "big", "serve", "coupled", "hydro",
                       "infer", "predict", "train"])
    if kind == "small":
        se = rng.choice([rng.randint(20, 70), rng.randint(300, 1000)])
        return dict(kind="query", nbox=rng.randint(1, 64), sizes="fixed",
                    natoms=rng.randint(256, 700), lo=0, hi=0, steps_equil=se,
                    steps_avg=rng.randint(20, 60) if se <= 70 else rng.randint(300, 1000))
    if kind == "one":
        return dict(kind="query", nbox=1, sizes="fixed", natoms=_log(rng, 769, 4096), lo=0, hi=0,
                    steps_equil=rng.randint(100, 1000), steps_avg=rng.randint(100, 1000))
    if kind == "uneven":
        return dict(kind="query", nbox=_log(rng, 100, 1024), sizes="fcc", natoms=0,
                    lo=rng.randint(3, 6), hi=rng.randint(7, 10),
                    steps_equil=rng.randint(200, 1000), steps_avg=rng.randint(200, 1000))
    if kind == "ragged":
        return dict(kind="query", nbox=_log(rng, 20, 304), sizes="log", natoms=0,
                    lo=rng.randint(40, 300), hi=rng.randint(700, 4096),
                    steps_equil=rng.randint(40, 200), steps_avg=rng.randint(40, 200))
    if kind == "big":
        return dict(kind="query", nbox=rng.randint(1, 3), sizes="fixed",
                    natoms=_log(rng, 4097, 32000), lo=0, hi=0,
                    steps_equil=rng.randint(40, 130), steps_avg=rng.randint(40, 130))
    if kind == "serve":
        return dict(kind="serve", nreq=_log(rng, 20, 304), lo=256, hi=_log(rng, 2000, 32000),
                    steps_equil=rng.randint(30, 100), steps_avg=rng.randint(30, 100))
    if kind == "coupled":
        return dict(kind="coupled", zones=_log(rng, 100, 2000), natoms=rng.randint(256, 500),
                    steps_equil=rng.randint(60, 200), steps_avg=rng.randint(100, 300),
                    first_equil=rng.randint(100, 600), first_avg=rng.randint(100, 300))
    if kind == "hydro":
        return dict(kind="hydro", zones=_log(rng, 100, 4000),
                    closure=rng.choice(["ideal", "mie"]), steps=rng.randint(20, 200))
    if kind == "infer":
        return dict(kind="infer", n=_log(rng, 1000, 1 << 20), chunk=_log(rng, 4096, 1 << 18))
    if kind == "predict":
        return dict(kind="predict", n=_log(rng, 100, 10000), chunk=rng.choice([1024, 4096, 65536]))
    return dict(kind="train", n=_log(rng, 4000, 32768), batch=rng.choice([256, 300, 512, 1024]),
                epochs=1)


# ---------------------------------------------------------------------------
# inputs

class _Held:
    """What a program keeps between calls; closed with it, the handle last."""

    def __init__(self, **kw):
        self.__dict__.update(kw)

    def __del__(self):
        for k in ("server", "hydro", "sg"):
            o = self.__dict__.pop(k, None)
            if o is not None:
                o.close()
        h = self.__dict__.pop("handle", None)
        if h is not None:
            m.mdeos_destroy(h)


_side_stream = None


def _stream():
    global _side_stream
    if _side_stream is None:
        _side_stream = torch.cuda.Stream()
    return _side_stream


def _requests(case, seed):
    """EOS requests (as the repository's workloads draw them) as a request array."""
    k = case["nbox"]
    rng = np.random.default_rng([20250806, seed])
    small = case["sizes"] == "fixed" and case["natoms"] < 769
    r_rng, t_rng = (RHO_SMALL, T_SMALL) if small else (RHO_UNEVEN, T_UNEVEN)
    if case["sizes"] == "fixed":
        n = np.full(k, case["natoms"])
    elif case["sizes"] == "fcc":
        n = 4 * rng.integers(case["lo"], case["hi"] + 1, k) ** 3
    else:
        n = np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"] + 1), k)).astype(np.int64)
    rho = rng.uniform(*r_rng, k)
    T = rng.uniform(*T_SMALL, k) if small else np.exp(rng.uniform(*np.log(t_rng), k))
    return _pack(n, rho, T, case, seed)


def _pack(n, rho, T, case, seed):
    a = np.zeros(len(n), dtype=m.REQUEST_DTYPE)
    a["rho"], a["natoms"] = rho, n
    a["e"] = (3.0 * n - 3.0) * T / (2.0 * n)   # the energy whose first temperature is T
    a["steps_equil"], a["steps_avg"] = case["steps_equil"], case["steps_avg"]
    a["seed"] = [W.box_seed(seed, i) for i in range(len(n))]
    a["element_id"] = np.arange(len(n))
    return a


def _params(seed, models=4):
    """Glorot-uniform weights of the ensemble, biases of a few per cent (FP32 vectors)."""
    rng = np.random.default_rng([7, seed])
    p = np.zeros((models, NPARAM), dtype=np.float32)
    l1, l2 = math.sqrt(6.0 / (H + 2)), math.sqrt(6.0 / (2 * H))
    for q in p:
        at = 0
        for size, lim in ((2 * H, l1), (H, 0.05), (H * H, l2), (H, 0.05), (H * H, l2), (H, 0.05),
                          (2 * H, l1), (2, 0.05)):
            q[at:at + size] = rng.uniform(-lim, lim, size)
            at += size
    return p


def _states(n, seed):
    """(rho, e) of n surrogate queries over the benchmark's range."""
    rng = np.random.default_rng([11, seed])
    return np.stack([rng.uniform(0.3, 1.2, n), rng.uniform(-5.0, 3.0, n)], axis=1)


def _answers(x, seed):
    """Training targets (P, T) with the shape of the LJ fluid's and its MD noise."""
    rng = np.random.default_rng([13, seed])
    rho, e = x[:, 0], x[:, 1]
    T = np.maximum((e + 6.0 * rho) / 1.5, 0.3)
    P = rho * T * (1.0 + rho + 2.0 * rho ** 3) - 6.0 * rho ** 2 + 4.0 * rho ** 5
    return np.stack([P, T], axis=1) * (1.0 + 0.005 * rng.standard_normal((len(x), 2)))


def _tube(case, seed):
    """Shock tube with states jittered by the seed: (x, u, rho, e)."""
    nz = case["zones"]
    rng = np.random.default_rng([17, seed])
    left = np.arange(nz) < nz // 2
    if case["closure"] == "mie":   # plate impact, copper (the hydro tests' constants)
        x = np.linspace(0.0, 0.001 * nz, nz + 1)
        u = np.where(np.arange(nz + 1) < nz // 3, 0.1 * rng.uniform(3.0, 6.9), 0.0)
        return x, u, 8.94 * rng.uniform(0.999, 1.001, nz), np.zeros(nz)
    x = np.linspace(0.0, 1.0, nz + 1)
    rho = np.where(left, 1.0, 0.125) * rng.uniform(0.98, 1.02, nz)
    p = np.where(left, 1.0, 0.1) * rng.uniform(0.98, 1.02, nz)
    return x, np.zeros(nz + 1), rho, p / ((5.0 / 3.0 - 1.0) * rho)


MIE = dict(mg_rho0=8.94, mg_c=0.3933, mg_s=1.5, mg_gamma=2.12)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "query":
        return _Held(kind=kind, handle=m.mdeos_create(), reqs=_requests(case, seed))
    if kind == "serve":
        k = case["nreq"]
        rng = np.random.default_rng([20250809, seed])
        n = np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), k)).astype(np.int64)
        reqs = _pack(n, rng.uniform(*RHO_UNEVEN, k), np.exp(rng.uniform(*np.log(T_UNEVEN), k)),
                     case, seed)
        reqs["element_id"] = 0
        h = m.mdeos_create()
        # 60 GB budget of the serving benchmark; the grid leaves the GPU soon after the
        # loop has drained (it shares it with the program's other work)
        srv = m.Server(h, hbm_budget_bytes=60 << 30, idle_ms=1)
        return _Held(kind=kind, handle=h, server=srv, reqs=reqs)
    if kind == "coupled":
        nz, n = case["zones"], case["natoms"]
        rng = np.random.default_rng([19, seed])
        left = np.arange(nz) < nz // 2
        rho = np.where(left, 1.0, 0.5) * rng.uniform(0.99, 1.01, nz)
        T0 = np.where(left, 2.0, 1.0) * rng.uniform(0.99, 1.01, nz)
        h = m.mdeos_create(m.mdeos_config_default(energy_ref_mode=m.MDEOS_REF_FIXED,
                                                  warm_slots=nz, warm_atoms=n))
        cfg = m.mdeos_hydro_config_default(
            nzones=nz, closure=m.CLOSURE_MD, natoms=n, steps_equil=case["steps_equil"],
            steps_avg=case["steps_avg"], steps_equil_first=case["first_equil"],
            steps_avg_first=case["first_avg"], first_temperature=1, e_ref=0.0,
            seed=20250807 + seed)
        hy = m.Hydro(h, cfg, np.linspace(0.0, float(nz), nz + 1), np.zeros(nz + 1), rho, T0)
        hy.step(1)   # the first step lifts every zone's box from the lattice
        return _Held(kind=kind, handle=h, hydro=hy)
    if kind == "hydro":
        x, u, rho, e = _tube(case, seed)
        h = m.mdeos_create()
        mie = case["closure"] == "mie"
        cfg = m.mdeos_hydro_config_default(
            nzones=case["zones"], closure=m.CLOSURE_MIE_GRUNEISEN if mie else m.CLOSURE_IDEAL_GAS,
            bc_left=m.BC_FREE if mie else m.BC_WALL, bc_right=m.BC_FREE if mie else m.BC_WALL,
            **(MIE if mie else {}))
        return _Held(kind=kind, handle=h, hydro=m.Hydro(h, cfg, x, u, rho, e),
                     steps=case["steps"])
    h = m.mdeos_create()
    if kind == "train":
        x = _states(case["n"], seed)
        sg = m.Surrogate(h, 4, case["batch"], seed=seed + 1)
        return _Held(kind=kind, handle=h, sg=sg, x=x, y=_answers(x, seed), batch=case["batch"],
                     epochs=case["epochs"], seed=seed)
    sg = m.Surrogate(h, 4, case["chunk"], seed=1)
    sg.set_params(_params(seed), np.array(NORM))
    x = _states(case["n"], seed)
    if kind == "predict":
        return _Held(kind=kind, handle=h, sg=sg, x=x)
    xd = torch.from_numpy(x).cuda()
    held = _Held(kind=kind, handle=h, sg=sg, x=xd, mean=torch.zeros_like(xd),
                 sd=torch.zeros_like(xd))
    torch.cuda.synchronize()
    return held


# ---------------------------------------------------------------------------
# one pass

def _fields(r):
    return {k: np.ascontiguousarray(r[k]).astype(np.int64) if r[k].dtype.kind == "u"
            else np.ascontiguousarray(r[k]) for k in r.dtype.names}


def run(s):
    if s.kind == "query":
        return _fields(m.mdeos_poll(s.handle, m.mdeos_submit(s.handle, s.reqs), len(s.reqs)))
    if s.kind == "serve":
        s.server.enqueue(s.reqs)
        got = s.server.wait_all(len(s.reqs))
        return _fields(got[np.argsort(got["id"])]["result"])   # ids ascend in request order
    if s.kind == "coupled":
        s.hydro.step(1)
        return {"hydro": s.hydro.state(), "eos": _fields(s.hydro.eos_results())}
    if s.kind == "hydro":
        s.hydro.step(s.steps)
        return s.hydro.state()
    if s.kind == "infer":
        s.sg.infer_device(s.x, s.mean, s.sd, stream=_stream())
        return {"mean": s.mean, "sd": s.sd}
    if s.kind == "predict":
        mean, sd, per_model = s.sg.predict(s.x, per_model=True)
        return {"mean": mean, "sd": sd, "per_model": per_model}
    loss = s.sg.train(s.x, s.y, s.epochs, batch=s.batch, lr=1e-3, seed=s.seed)
    params, norm = s.sg.get_params()
    return {"loss": loss, "params": params, "norm": norm}


# ---------------------------------------------------------------------------
# what a pass cannot do without

def _md_flops(atoms, rho, steps):
    """In-cutoff pairs (each once) at the mean density, 27 flop each, every step."""
    return 27.0 * 0.5 * atoms * rho * 4.0 / 3.0 * math.pi * 2.5 ** 3 * steps


def work(case):
    kind = case["kind"]
    steps = case.get("steps_equil", 0) + case.get("steps_avg", 0)
    if kind == "query":
        k = case["nbox"]
        if case["sizes"] == "fixed":
            atoms = k * case["natoms"]
        elif case["sizes"] == "fcc":
            side = range(case["lo"], case["hi"] + 1)
            atoms = k * sum(4 * c ** 3 for c in side) / len(side)
        else:
            atoms = k * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        return {"bytes": k * (72 + 200), "flops": _md_flops(atoms, 0.75, steps)}
    if kind == "serve":
        k = case["nreq"]
        atoms = k * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        return {"bytes": k * (72 + 200), "flops": _md_flops(atoms, 0.75, steps)}
    if kind == "coupled":
        atoms = case["zones"] * case["natoms"]   # states read and written once: 32 B per atom
        return {"bytes": 64.0 * atoms + case["zones"] * (200 + 11 * 8),
                "flops": _md_flops(atoms, 0.75, steps)}
    if kind == "hydro":
        return {"bytes": 88.0 * case["zones"], "flops": 60.0 * case["zones"] * case["steps"]}
    mac = 2 * H + 2 * H * H + 2 * H
    if kind in ("infer", "predict"):
        per_model = 32 if kind == "predict" else 0
        return {"bytes": case["n"] * (48.0 + per_model) + 4 * NPARAM * 4,
                "flops": 8.0 * mac * case["n"]}
    done = case["n"] // case["batch"] * case["batch"] * case["epochs"]
    return {"bytes": 32.0 * done + 4 * NPARAM * 4 * 7, "flops": 3 * 8.0 * mac * done}


# ---------------------------------------------------------------------------
# the same in 64 bits

def exact(case, seed):
    kind = case["kind"]
    if kind == "query":
        # trajectories stay comparable over some hundred steps; the minimum image needs
        # L >= 2 r_c
        if (case["sizes"] != "fixed" or not 256 <= case["natoms"] <= 768 or case["nbox"] > 64
                or case["steps_equil"] + case["steps_avg"] > 130):
            return None
        rs = [_exact_query(q) for q in _requests(case, seed)]
        return {k: np.array([r[k] for r in rs]) if rs[0][k] is not None else None for k in rs[0]}
    if kind == "hydro":
        return _exact_hydro(case, seed)
    if kind in ("infer", "predict"):
        return _exact_predict(case, seed)
    return None   # trajectories, and training steps that divide by a gradient's size


def _philox(seed, n):
    """Philox4x32-10 of counters (atom, 0, 0, 0) under the 64-bit key `seed`."""
    mask = np.uint64(0xFFFFFFFF)
    c = [np.arange(n, dtype=np.uint64)] + [np.zeros(n, dtype=np.uint64)] * 3
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        a, b = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(b >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), b & mask,
             (a >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), a & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return [(v.astype(np.float64) + 0.5) * 2.0 ** -32 for v in c]


def _exact_query(q, rc=2.5, dt=0.005, blocks=10, every=10):
    """One EOS query in FP64: lifting, two NVE segments, thermostatted averaging."""
    n, rho, se, sa = int(q["natoms"]), float(q["rho"]), int(q["steps_equil"]), int(q["steps_avg"])
    L = float(np.float32((n / rho) ** (1.0 / 3.0)))
    ndof, V = 3.0 * n - 3.0, L ** 3
    nc = 1
    while 4 * nc ** 3 < n:
        nc += 1
    i = np.arange(n)
    c, b = i >> 2, i & 3
    x = np.stack([(c % nc + 0.5 * np.isin(b, (1, 2))), (c // nc % nc + 0.5 * np.isin(b, (1, 3))),
                  (c // nc ** 2 + 0.5 * np.isin(b, (2, 3)))], axis=1) * (L / nc)
    x = torch.from_numpy(x).cuda()
    eye = torch.eye(n, dtype=torch.bool, device="cuda")
    ucut = 4.0 * (rc ** -12 - rc ** -6)

    def forces(x):
        d = x[:, None, :] - x[None, :, :]
        d = d - L * torch.round(d / L)
        r2 = (d * d).sum(-1)
        on = (r2 < rc * rc) & ~eye
        i2 = torch.where(on, 1.0 / torch.where(on, r2, 1.0), 0.0)
        s6 = i2 ** 3
        fr = 24.0 * s6 * (2.0 * s6 - 1.0) * i2
        f = (fr[:, :, None] * d).sum(1)
        e = 0.5 * torch.where(on, 4.0 * s6 * (s6 - 1.0) - ucut, 0.0).sum()
        w = 0.5 * torch.einsum("ij,ija,ijb->ab", fr, d, d)
        return f, float(e), w.cpu().numpy(), int(on.sum())

    f, e_cold, _, _ = forces(x)
    e_tgt = n * float(q["e"]) + e_cold
    Tk = 2.0 * (e_tgt - e_cold) / ndof
    u = _philox(int(q["seed"]), n)
    r01, r23 = np.sqrt(-2.0 * np.log(u[0])), np.sqrt(-2.0 * np.log(u[2]))
    v = math.sqrt(Tk) * np.stack([r01 * np.cos(2 * np.pi * u[1]), r01 * np.sin(2 * np.pi * u[1]),
                                  r23 * np.cos(2 * np.pi * u[3])], axis=1)
    v -= v.mean(0)
    v *= math.sqrt(Tk * ndof / (v * v).sum())
    v = torch.from_numpy(v).cuda()
    lam, seg, pos, base = 1.0, 0, 0, se // 2
    length, ebar = base, []
    S, ep, ek, Ps, Ts, pairs = np.zeros((3, 3)), [], [], [], [], []
    for step in range(se + sa):
        v = lam * v + 0.5 * dt * f
        x = x + dt * v
        f, e, w, npair = forces(x)
        v = v + 0.5 * dt * f
        k = (v.T @ v).cpu().numpy()
        Ti, lam = float(np.trace(k)) / ndof, 1.0
        if step < se:
            if pos >= length - max(1, (length + 9) // 10):
                ebar.append(e)
            pos += 1
            if pos == length:
                Tk = 2.0 * (e_tgt - float(np.mean(ebar))) / ndof
                lam, ebar, pos, seg = math.sqrt(Tk / Ti), [], 0, seg + 1
                length = base + se % 2 if seg == 1 else base
            continue
        S += (k + w) / V
        ep.append(e)
        ek.append(0.5 * float(np.trace(k)))
        Ps.append(float(np.trace(k + w)) / (3.0 * V))
        Ts.append(Ti)
        pairs.append(npair)
        if (step - se + 1) % every == 0:
            lam = math.sqrt(Tk / Ti)
    S /= sa
    blk = np.arange(sa) * blocks // sa

    def se_of(a):
        means = np.array([np.mean(np.array(a)[blk == k]) for k in range(blocks)])
        return math.sqrt(((means - means.mean()) ** 2).sum() / (blocks - 1) / blocks)

    return {"P": np.mean(Ps), "T": np.mean(Ts),
            "sigma": np.array([S[0, 0], S[1, 1], S[2, 2], S[0, 1], S[0, 2], S[1, 2]]),
            "epot": np.mean(ep) / n, "ekin": np.mean(ek) / n,
            "e_achieved": (np.mean(ep) + np.mean(ek) - e_cold) / n, "P_se": se_of(Ps),
            "T_se": se_of(Ts), "T_target": Tk, "e_cold": e_cold / n, "L": L,
            "pairs_per_step": np.mean(pairs),
            # how the list was kept, and tags
            "cand_per_step": None, "element_id": None, "natoms": None, "status": None,
            "nlist_builds": None, "path": None, "warm": None, "nlist_retries": None}


def _exact_hydro(case, seed):
    x, u, rho, e = _tube(case, seed)
    mie = case["closure"] == "mie"
    g = 5.0 / 3.0
    mz = rho * np.diff(x)
    M = np.r_[0.5 * mz, 0.0] + np.r_[0.0, 0.5 * mz]
    if not mie:
        u[0] = u[-1] = 0.0
    t, prev = 0.0, 0.0
    for _ in range(case["steps"]):
        if mie:
            r0, C, s, G = MIE["mg_rho0"], MIE["mg_c"], MIE["mg_s"], MIE["mg_gamma"]
            eta = 1.0 - r0 / rho
            den = 1.0 - s * eta
            PH = r0 * C * C * eta / den ** 2
            EH = PH * eta / (2.0 * r0)
            P = PH + G * rho * (e - EH)
            dPH = r0 * C * C * (1.0 + s * eta) / den ** 3
            dEH = (PH + eta * dPH) / (2.0 * r0)
            c2 = (dPH - G * rho * dEH) * r0 / rho ** 2 + G * (e - EH) + P / rho ** 2 * (G * rho)
        else:
            P = (g - 1.0) * rho * e
            c2 = g * P / rho
        c, du, dx = np.sqrt(c2), np.diff(u), np.diff(x)
        q = np.where(du < 0.0, rho * (2.0 * du * du - 0.5 * c * du), 0.0)
        dt = 0.5 * np.min(dx / (c + 4.0 * np.maximum(-du, 0.0)))
        dt = min(dt, 1.1 * prev) if prev > 0.0 else dt
        Pq = P + q
        un = u + dt * (np.r_[0.0, Pq] - np.r_[Pq, 0.0]) / M
        if not mie:
            un[0] = un[-1] = 0.0
        uh = 0.5 * (u + un)
        u, x = un, x + dt * uh
        e = e - dt * Pq * np.diff(uh) / mz
        rho = mz / np.diff(x)
        t, prev = t + dt, dt
    return {"x": x, "u": u, "rho": rho, "e": e, "P": P, "q": q, "c2": c2, "t": t, "dt": prev,
            "steps": None}


def _exact_predict(case, seed):
    x = torch.from_numpy(_states(case["n"], seed)).cuda()
    nm = NORM
    x = (x - x.new_tensor(nm[:2])) / x.new_tensor(nm[2:4])
    ys = []
    for p in torch.from_numpy(_params(seed)).cuda().double():
        at, w = 0, []
        for rows, cols in ((H, 2), (H, 1), (H, H), (H, 1), (H, H), (H, 1), (2, H), (2, 1)):
            w.append(p[at:at + rows * cols].reshape(rows, cols))
            at += rows * cols
        h = x
        for k in (0, 2, 4):
            h = torch.tanh(h @ w[k].T + w[k + 1].T)
        ys.append(h @ w[6].T + w[7].T)
    y = torch.stack(ys)
    phys = y * x.new_tensor(nm[6:8]) + x.new_tensor(nm[4:6])
    out = {"mean": phys.mean(0), "sd": phys.std(0, unbiased=False)}
    if case["kind"] == "predict":
        out["per_model"] = y
    return out
