"""Performance cases of libnbody: what its users' programs have it do.

A case is a dict of plain values; ``prepare`` loads a system and ``run``
makes one pass through the public calls (``include/nbody.h`` by way of
``paper_1104_2700_gb300.nbody``).  Four kinds:

``force``     a host integrator's call: predict every particle to the block
              time, then acc, jerk and pot of one block (device arrays).
``static``    the allocation-free force call on the caller's device arrays.
``steps``     an integration with outputs: from a stored state, integrate to
              each output time in turn, the state read into device arrays.
``ensemble``  the same for independent systems advanced together.

Systems are Plummer models in N-body units with the softening eps = 4 / N
unless the case says otherwise; a block's members are drawn with weights
that fall with radius, as short timesteps do.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1104_2700_gb300 import ics, nbody

ETA = 0.02
ETA_START = 0.01
DT_MAX = 1.0 / 16
T_BLOCK = 2.0 ** -12  # block time of the force cases
PAIR_FLOPS = 60       # acc + jerk + pot of one pair, the paper's convention


def listed():
    return [
        # the smallest call: one short-step block of the paper's mid-size model
        {"name": "force hybrid 16384/32", "kind": "force", "precision": "hybrid", "n": 16384,
         "n_act": 32, "salpeter": False},
        # a middling block of a large model, ragged in both sizes
        {"name": "force hybrid 65521/1999", "kind": "force", "precision": "hybrid", "n": 65521,
         "n_act": 1999, "salpeter": False},
        # every particle of the large model: the synchronised blocks, the
        # roofline workload
        {"name": "force hybrid 65536/all", "kind": "force", "precision": "hybrid", "n": 65536,
         "n_act": 65536, "salpeter": False},
        # a stellar mass function, a block of a few hundred stars
        {"name": "force hybrid salpeter 32003/300", "kind": "force", "precision": "hybrid",
         "n": 32003, "n_act": 300, "salpeter": True},
        # the paper's mixed scheme as a plain force library, ragged
        {"name": "force mixed 30011/all", "kind": "force", "precision": "mixed", "n": 30011,
         "n_act": 30011, "salpeter": False},
        # double-single forces of a whole model (reference-quality forces)
        {"name": "force ds 16384/all", "kind": "force", "precision": "ds", "n": 16384,
         "n_act": 16384, "salpeter": False},
        # the all-FP64 path (energies and baselines run it), ragged
        {"name": "force fp64 4099/all", "kind": "force", "precision": "fp64", "n": 4099,
         "n_act": 4099, "salpeter": False},
        # the allocation-free call on a block of a host framework's particles
        {"name": "static 8192/500", "kind": "static", "precision": "ds", "n": 8192,
         "n_act": 500, "salpeter": False},
        # the paper's small integration: launches and latency per block step
        {"name": "steps hybrid 1024", "kind": "steps", "precision": "hybrid", "n": 1024,
         "eps": 1.0 / 64, "outputs": 2, "log2_dt_out": -6},
        # a mid-size integration between two close outputs
        {"name": "steps hybrid 16384", "kind": "steps", "precision": "hybrid", "n": 16384,
         "eps": 4.0 / 16384, "outputs": 1, "log2_dt_out": -7},
        # the same loop in double-single, an odd size
        {"name": "steps ds 4001", "kind": "steps", "precision": "ds", "n": 4001,
         "eps": 4.0 / 4001, "outputs": 1, "log2_dt_out": -7},
        # many clusters of uneven size advanced together
        {"name": "ensemble hybrid 48", "kind": "ensemble", "precision": "hybrid", "k": 48,
         "size_seed": 4, "n_lo": 256, "n_hi": 4096, "outputs": 1, "log2_dt_out": -8},
    ]


# Largest pair count of one force call by precision (about the same time), so
# that no drawn case costs more than the listed ones.
MAX_PAIRS = {"hybrid": 65536 ** 2, "mixed": 65536 ** 2, "ds": 16384 ** 2, "fp64": 8192 ** 2}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["force", "force", "force", "steps", "ensemble", "static"])
    if kind == "steps":
        precision = rng.choice(["hybrid", "hybrid", "ds", "fp64"])
        n = _log_int(rng, 256, {"hybrid": 16384, "ds": 8192, "fp64": 2048}[precision])
        return {"kind": kind, "precision": precision, "n": n,
                "eps": rng.choice([4.0 / n, 1.0 / 64]), "outputs": rng.randint(1, 3),
                "log2_dt_out": -9 if n > 4096 else -8}
    if kind == "ensemble":
        return {"kind": kind, "precision": rng.choice(["hybrid", "hybrid", "ds"]),
                "k": _log_int(rng, 4, 64), "size_seed": rng.randrange(1 << 20), "n_lo": 256,
                "n_hi": rng.choice([1024, 2048, 4096]), "outputs": 1,
                "log2_dt_out": rng.choice([-10, -9])}
    if kind == "static":
        precision = "ds"
        n = _log_int(rng, 256, 16384)
    else:
        precision = rng.choice(["hybrid", "hybrid", "mixed", "ds", "fp64"])
        n = _log_int(rng, 256, {"hybrid": 65536, "mixed": 65536, "ds": 32768, "fp64": 16384}[precision])
    most = min(n, MAX_PAIRS[precision] // n)
    n_act = most if rng.random() < 0.25 else _log_int(rng, 1, most)
    return {"kind": kind, "precision": precision, "n": n, "n_act": n_act,
            "salpeter": rng.random() < 0.25}


# --- inputs --------------------------------------------------------------------
def _system(case, seed):
    """m, r, v, eps of a force or static case and its block."""
    n, n_act = case["n"], case["n_act"]
    masses = ics.salpeter_masses(n, seed) if case["salpeter"] else None
    m, r, v = ics.plummer(n, seed, masses=masses)
    if n_act == n:
        idx = np.arange(n, dtype=np.int32)
    else:
        # sampling without replacement, weights (1 + r^2 / a^2)^(-5/4): the
        # square root of the Plummer density, as free-fall times go
        g = np.random.RandomState(seed & 0x7FFFFFFF)
        w = -1.25 * np.log1p(np.einsum("ij,ij->i", r, r) / 0.3468)
        idx = np.sort(np.argsort(-(w + g.gumbel(size=n)), kind="stable")[:n_act]).astype(np.int32)
    return m, r, v, 4.0 / n, idx


def _ensemble(case, seed):
    return ics.ensemble(case["k"], case["size_seed"], seed, case["n_lo"], case["n_hi"])[1:]


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _rows(n):
    return [torch.empty((n, 3), dtype=torch.float64, device="cuda") for _ in range(2)] + \
        [torch.empty(n, dtype=torch.float64, device="cuda")]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("force", "static"):
        m, r, v, eps, idx = _system(case, seed)
        s = {"kind": kind, "idx": _cuda(idx), "out": _rows(len(idx))}
        if kind == "static":
            s.update(m=_cuda(m), r=_cuda(r), v=_cuda(v), eps=eps)
            return s
        ctx = nbody.Context(case["precision"], eta_start=ETA_START, dt_max=DT_MAX)
        ctx.set_particles(m, r, v, eps, ETA)
        s["ctx"] = ctx
        return s
    ctx = nbody.Context(case["precision"], eta_start=ETA_START, dt_max=DT_MAX)
    if kind == "steps":
        m, r, v = ics.plummer(case["n"], seed)
        ctx.set_particles(m, r, v, case["eps"], ETA)
    else:
        off, m, r, v, eps = _ensemble(case, seed)
        ctx.set_ensemble(off, m, r, v, eps, ETA)
    snap = torch.empty(ctx.snapshot_bytes() // 8 + 1, dtype=torch.float64, device="cuda")
    ctx.snapshot(snap)
    n = ctx.n
    out = [torch.empty((n, 3), dtype=torch.float64, device="cuda") for _ in range(4)] + \
        [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2)]
    return {"kind": kind, "ctx": ctx, "snap": snap, "out": out,
            "times": [(k + 1) * 2.0 ** case["log2_dt_out"] for k in range(case["outputs"])]}


# --- one pass ------------------------------------------------------------------
def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _check(st):
    if st != nbody.NB_OK:
        raise RuntimeError(nbody.nb_status_string(st))


def run(s):
    if s["kind"] == "force":
        ctx = s["ctx"]
        ctx.predict(T_BLOCK)
        return list(ctx.force(s["idx"], *s["out"]))
    if s["kind"] == "static":
        acc, jerk, pot = s["out"]
        _check(nbody.nb_force_static(s["m"].numel(), _p(s["m"]), _p(s["r"]), _p(s["v"]), s["eps"],
                                     1.0, s["idx"].numel(), _p(s["idx"]), _p(acc), _p(jerk),
                                     _p(pot), None))
        return [acc, jerk, pot]
    ctx = s["ctx"]
    ctx.restore(s["snap"])
    for t in s["times"]:
        ctx.step_until(t)
    _check(nbody.nb_get_state(ctx.handle, *[_p(x) for x in s["out"]], 1))
    return s["out"]


# --- what a pass cannot do without -----------------------------------------------
def _integration_work(n, span):
    """Bytes and flops of integrating n particles over a time span: about
    930 (n / 1024)^0.27 steps per particle and unit time, in blocks of about
    0.4 n^(2/3) members; each block reads every particle's state once."""
    steps = max(n, n * 930.0 * (n / 1024.0) ** 0.27 * span)
    blocks = steps / (0.4 * n ** (2.0 / 3.0))
    return blocks * n * 112.0 + steps * 200.0, steps * n * PAIR_FLOPS


def work(case):
    if case["kind"] in ("force", "static"):
        state = 56 if case["kind"] == "static" else 112  # bytes of one particle's inputs
        return {"bytes": case["n"] * state + case["n_act"] * 60,
                "flops": PAIR_FLOPS * case["n"] * case["n_act"]}
    span = case["outputs"] * 2.0 ** case["log2_dt_out"]
    if case["kind"] == "steps":
        b, f = _integration_work(case["n"], span)
        return {"bytes": b, "flops": f}
    sizes = ics.ensemble_sizes(case["k"], case["size_seed"], case["n_lo"], case["n_hi"])
    parts = [_integration_work(float(x), span) for x in sizes]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# --- the same in plain 64-bit torch --------------------------------------------------
def _force64(m, r, v, rp, vp, idx, eps):
    """acc, jerk, pot of rows (rp, vp)[idx] from all (rp, vp), 64 bits."""
    n = len(m)
    acc = torch.empty((len(idx), 3), dtype=torch.float64, device=m.device)
    jerk = torch.empty_like(acc)
    pot = torch.empty(len(idx), dtype=torch.float64, device=m.device)
    x, u = rp.t().contiguous(), vp.t().contiguous()
    step = max(1, (1 << 24) // n)
    for a in range(0, len(idx), step):
        i = idx[a:a + step]
        d = [x[c][None, :] - rp[i, c][:, None] for c in range(3)]
        w = [u[c][None, :] - vp[i, c][:, None] for c in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps
        me = torch.arange(len(i), device=m.device)
        r2[me, i] = math.inf  # no self pair
        ri = r2.rsqrt_()
        mr = m[None, :] * ri
        pot[a:a + step] = -mr.sum(1)
        ri.mul_(ri)
        g = mr.mul_(ri)
        t = (d[0] * w[0] + d[1] * w[1] + d[2] * w[2]).mul_(ri).mul_(-3.0)
        for c in range(3):
            acc[a:a + step, c] = (g * d[c]).sum(1)
            jerk[a:a + step, c] = (g * (w[c] + t * d[c])).sum(1)
    return acc, jerk, pot


def _norm(x):
    return x.square().sum(1).sqrt()


def _pow2_floor(x):
    return torch.ldexp(torch.ones_like(x), torch.frexp(x)[1] - 1)


def _predict64(s, t):
    h = (t - s["t"])[:, None]
    rp = s["r"] + h * (s["v"] + h * (0.5 * s["a"] + h * s["j"] / 6.0))
    vp = s["v"] + h * (s["a"] + h * (0.5 * s["j"]))
    return rp, vp


def _load64(m, r, v, eps):
    m, r, v = (torch.from_numpy(np.array(x)).to("cuda" if torch.cuda.is_available() else "cpu")
               for x in (m, r, v))
    every = torch.arange(len(m), device=m.device)
    a, j, _ = _force64(m, r, v, r, v, every, eps)
    na, nj = _norm(a), _norm(j)
    dt = _pow2_floor(torch.clamp(ETA_START * na / nj, max=DT_MAX))  # j = 0: inf, so dt_max
    return {"m": m, "r": r, "v": v, "a": a, "j": j, "t": torch.zeros_like(m), "dt": dt}


def _integrate64(s, eps, t_end):
    """The fourth-order Hermite scheme with block timesteps to t_end."""
    while True:
        nxt = s["t"] + s["dt"]
        t = float(nxt.min())
        if t > t_end:
            return
        i = (nxt == t).nonzero()[:, 0]
        rp, vp = _predict64(s, t)
        a1, j1, _ = _force64(s["m"], s["r"], s["v"], rp, vp, i, eps)
        h = s["dt"][i]
        hc = h[:, None]
        a0, j0 = s["a"][i], s["j"][i]
        da = a0 - a1
        sn = 2.0 * (-3.0 * da - hc * (2.0 * j0 + j1)) / hc ** 2
        cr = 6.0 * (2.0 * da + hc * (j0 + j1)) / hc ** 3
        s["r"][i] = rp[i] + hc ** 4 * (sn / 24.0 + hc * cr / 120.0)
        s["v"][i] = vp[i] + hc ** 3 * (sn / 6.0 + hc * cr / 24.0)
        s["a"][i], s["j"][i], s["t"][i] = a1, j1, t
        A, J, S, C = _norm(a1), _norm(j1), _norm(sn + hc * cr), _norm(cr)
        cand = torch.clamp(ETA * torch.sqrt((A * S + J * J) / (J * C + S * S)), max=DT_MAX)
        cand = torch.where(torch.isnan(cand), torch.full_like(cand, DT_MAX), cand)
        k = t / (2.0 * h)
        up = (cand >= 2.0 * h) & (k == torch.round(k))
        down = torch.minimum(h, _pow2_floor(cand))
        s["dt"][i] = torch.where(up, 2.0 * h, torch.where(cand >= h, h, down))


def exact(case, seed):
    if case["kind"] in ("force", "static"):
        m, r, v, eps, idx = _system(case, seed)
        if case["kind"] == "static":
            m, r, v, i = (_cuda(x) if torch.cuda.is_available() else torch.from_numpy(x)
                          for x in (m, r, v, idx))
            return list(_force64(m, r, v, r, v, i.long(), eps))
        s = _load64(m, r, v, eps)
        rp, vp = _predict64(s, T_BLOCK)
        i = torch.from_numpy(idx).long().to(rp.device)
        return list(_force64(s["m"], s["r"], s["v"], rp, vp, i, eps))
    t_end = case["outputs"] * 2.0 ** case["log2_dt_out"]
    if case["kind"] == "steps":
        systems = [(*ics.plummer(case["n"], seed), case["eps"])]
    else:
        if case["k"] > 16:
            return None  # one plain integration after another: minutes
        off, m, r, v, eps = _ensemble(case, seed)
        systems = [(m[a:b], r[a:b], v[a:b], eps[q])
                   for q, (a, b) in enumerate(zip(off[:-1], off[1:]))]
    done = []
    for m, r, v, eps in systems:
        s = _load64(m, r, v, float(eps))
        _integrate64(s, float(eps), t_end)
        done.append(s)
    return [torch.cat([s[q] for s in done]) for q in ("r", "v", "a", "j", "t", "dt")]
