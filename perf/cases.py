"""The work that this framework is used for, as cases that can be timed and compared.

Lennard-Jones clusters (and their Morse twins) go through the three public entry points:

* eval:  lj_energy_grad_batched -- energies and gradients of a batch, the call that a user's own
         optimiser, sampler or trainer makes; uniform and uneven batches, FP32 and FP64, both
         potentials, one configuration at a time or tens of thousands;
* min:   lbfgs_minimize_batched -- the quench of a batch of displaced clusters;
* bh:    bh_step_batched -- Basin Hopping steps of independent walkers, K candidates each.

Structures are Mackay icosahedra with a partial outer layer up to 309 atoms (the motif of the
small clusters' minima) and fcc fragments above, displaced by Gaussian jitter.  The quenches and
the Basin Hopping moves are displacements from which a cluster falls back into the minimum that
it came from, as late in a search: from the violent starts of its beginning a descent ends in one
of thousands of minima, and which one is decided by the last bit of its first steps.

What run() returns: energies, gradients, status, the walkers' whole state and the step trace.
A minimum's position and orientation in space are an artefact of the path that led to it (nothing
in the energy holds them), and of K candidates that fell into one minimum an energy difference of
1e-13 picks the one that is kept; so minimised structures leave in internal coordinates, the
distances of every atom to the first four, which are all of a structure but that rigid motion.
The stopping rule ||g||_inf < 1e-6 fixes distances to about that, so they are FP32.  An evaluation
in FP32 arithmetic is handed on in FP32, its energies too.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2510_25938_gb300 import inputs as I
from paper_2510_25938_gb300 import lj_bh as L

ICO_MAX = 309                      # atoms of the icosahedron of four shells
MORSE_RHO = 6.0


def listed():
    return [
        # a user's own optimiser asks for one cluster at a time: all launch and latency
        dict(name="eval-one-lj38-f64", op="eval", n=38, cand=1, prec="f64", pot="lj"),
        # the evaluation benchmark of this repository: 65,536 configurations of LJ38
        dict(name="eval-lj38-f32", op="eval", n=38, cand=65536, prec="f32", pot="lj"),
        dict(name="eval-lj38-f64", op="eval", n=38, cand=65536, prec="f64", pot="lj"),
        # a library of clusters of all sizes, rescored in one call (sizes 13..150)
        dict(name="eval-uneven-f32", op="eval", n=150, n_lo=13, cand=4096, prec="f32", pot="lj"),
        # the same benchmark on the other pair potential
        dict(name="eval-morse38-f32", op="eval", n=38, cand=65536, prec="f32", pot="morse"),
        # the large clusters: forces for a batch of fcc fragments
        dict(name="eval-fcc500-f32", op="eval", n=500, cand=1024, prec="f32", pot="lj"),
        dict(name="eval-fcc1000-f64", op="eval", n=1000, cand=256, prec="f64", pot="lj"),
        # quenching a set of displaced LJ38 clusters, as after a molecular-dynamics run
        dict(name="min-lj38-mixed", op="min", n=38, cand=4096, prec="mixed", pot="lj", m=10,
             jitter=0.04, switch=1e-4, gtol=1e-6),
        # the uneven batch of this repository's benchmark (4,096 clusters of 13..150 atoms)
        dict(name="min-uneven-mixed", op="min", n=150, n_lo=13, cand=4096, prec="mixed",
             pot="lj", m=10, jitter=0.04, switch=0.0, gtol=1e-6),
        # its large clusters (fcc fragments of 500 atoms, m = 20)
        dict(name="min-fcc500-mixed", op="min", n=500, cand=1024, prec="mixed", pot="lj", m=20,
             jitter=0.1, switch=1e-4, gtol=1e-6),
        # the headline: 64 walkers x 8 candidates of LJ38, 25 steps a launch, late in a search
        dict(name="bh-lj38-mixed", op="bh", n=38, walkers=64, K=8, steps=25, prec="mixed",
             pot="lj", step=0.1, switch=1e-4),
        # the plain sequential search: one walker, one candidate, LJ13, FP64 throughout
        dict(name="bh-lj13-f64", op="bh", n=13, walkers=1, K=1, steps=50, prec="f64", pot="lj",
             step=0.15, switch=0.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["eval", "eval", "eval", "min", "min", "bh"])
    pot = "morse" if rng.random() < 0.25 else "lj"
    if op == "eval":
        prec = rng.choice(["f32", "f64"])
        n = _log_int(rng, 3, 1024)
        # up to the pairs of the largest listed evaluation of that precision
        most = (1.0e8 if prec == "f32" else 4.0e7) / (n * n)
        c = dict(op=op, n=n, cand=_log_int(rng, 1, max(2, min(65536, most))), prec=prec, pot=pot)
        if rng.random() < 0.35 and n > 4:
            c["n_lo"] = rng.randint(2, n // 2)
        return c
    if op == "min":
        # FP64 to scipy's L-BFGS-B default tolerance: 1e-6 is at the noise of an FP64 energy
        prec = rng.choice(["mixed", "mixed", "f64"])
        n = _log_int(rng, 13, 500 if prec == "mixed" else 150)
        n = _UNSTABLE.get(n, n)
        most = (4.0e7 if prec == "mixed" else 4.0e6) / (n * n)
        c = dict(op=op, n=n, cand=_log_int(rng, 1, max(2, min(4096, most))), prec=prec, pot=pot,
                 m=rng.choice([5, 10, 10, 20]), jitter=0.04,
                 switch=rng.choice([0.0, 1e-4]) if prec == "mixed" else 0.0,
                 gtol=1e-6 if prec == "mixed" else 1e-5)
        if rng.random() < 0.35 and n > 30:
            c["n_lo"] = rng.randint(13, n // 2)
        return c
    prec = rng.choice(["mixed", "mixed", "f64"])
    n = _log_int(rng, 13, 150)
    n = _UNSTABLE.get(n, n)
    K = rng.choice([1, 2, 4, 8, 8, 16])
    w = _log_int(rng, 1, 64)
    most = 25 if prec == "mixed" and n <= 64 else 6
    return dict(op=op, n=n, walkers=w, K=K, steps=rng.randint(2, most), prec=prec, pot=pot,
                step=0.08, switch=1e-4 if prec == "mixed" else 0.0)


# ---------------------------------------------------------------------------
# structures
# ---------------------------------------------------------------------------
def _mackay(shells):
    """Sites of the Mackay icosahedron and the shell that each is on."""
    phi = (1 + 5 ** 0.5) / 2
    v = np.array([(0, a, b * phi) for a in (1, -1) for b in (1, -1)])
    v = np.concatenate([v, v[:, [1, 2, 0]], v[:, [2, 0, 1]]])
    near = np.abs(np.linalg.norm(v[:, None] - v[None], axis=-1) - 2) < 1e-6
    faces = [f for f in itertools.combinations(range(12), 3)
             if near[f[0], f[1]] and near[f[0], f[2]] and near[f[1], f[2]]]
    pts, shell = [np.zeros((1, 3))], [0]
    for k in range(1, shells + 1):
        p = np.array([v[a] * i + v[b] * j + v[c] * (k - i - j) for a, b, c in faces
                      for i in range(k + 1) for j in range(k + 1 - i)])
        p = np.unique(np.round(p, 9), axis=0)
        pts.append(p)
        shell += [k] * len(p)
    return np.concatenate(pts), np.array(shell)


_SITES = _mackay(4)
# a few atoms on a closed layer have no place of their own: the next size that is a minimum
_UNSTABLE = {14: 18, 15: 18, 16: 18, 17: 18, 56: 59, 57: 59, 58: 59, 61: 62, 148: 149}


def _structure(n):
    """(n, 3): an icosahedron whose outer shell is filled from one side, or an fcc fragment."""
    if n > ICO_MAX:
        return I.fcc_sites(n)
    p, shell = _SITES
    r = np.linalg.norm(p, axis=1)
    side = p @ np.array([0.3, 0.5, 0.81]) / np.maximum(r, 1e-9)
    order = np.lexsort((-side, shell))
    return p[order[:n]] * (1.06 / r[1])


def _sizes(case):
    """Atoms of each candidate of an uneven batch, or None; the same for every seed."""
    if "n_lo" not in case:
        return None
    sizes = I.uneven_sizes(case["cand"], case["n_lo"], case["n"], I.workload_seed(3))
    if case["op"] == "min":
        sizes = np.array([min(_UNSTABLE.get(int(k), int(k)), case["n"]) for k in sizes])
    return sizes


def _base(case):
    """The undisplaced atoms of the batch, packed (total, 3), and its offsets (or None)."""
    sizes = _sizes(case)
    if sizes is None:
        one = torch.as_tensor(_structure(case["n"]), device="cuda")
        return one.repeat(case.get("cand", 1), 1), None
    by_size = {int(k): _structure(int(k)) for k in np.unique(sizes)}
    x = np.concatenate([by_size[int(k)] for k in sizes])
    return torch.as_tensor(x, device="cuda"), I.offsets_from_sizes(sizes)


def _displaced(case, seed):
    x, off = _base(case)
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = x + case.get("jitter", 0.05) * torch.randn(x.shape, generator=g, device="cuda",
                                                   dtype=torch.float64)
    return x.reshape(-1).contiguous(), off


def _pot(case):
    return dict(potential=L.LJ_POT_MORSE if case["pot"] == "morse" else L.LJ_POT_LJ,
                rho=MORSE_RHO)


def _params(case):
    return L.LbfgsParams(m=case.get("m", 10), gtol=case.get("gtol", 1e-6),
                         prec=L.LJ_PREC_MIXED if case["prec"] == "mixed" else L.LJ_PREC_FP64,
                         switch_gtol=case["switch"], **_pot(case))


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def prepare(case, seed):
    ctx = L.Ctx()
    s = dict(case=case, ctx=ctx)
    if case["op"] == "bh":
        n, w = case["n"], case["walkers"]
        x, e = _relaxed(n, case["pot"])
        x = x.reshape(1, -1).repeat(w, 1)
        s["start"] = dict(x_cur=x, e_cur=torch.full((w,), e, device="cuda", dtype=torch.float64),
                          x_best=x.clone(),
                          e_best=torch.full((w,), e, device="cuda", dtype=torch.float64),
                          stepsize=torch.full((w,), case["step"], device="cuda",
                                              dtype=torch.float64),
                          win_accept=torch.zeros(w, dtype=torch.int32, device="cuda"),
                          n_accept=torch.zeros(w, dtype=torch.int32, device="cuda"))
        s["state"] = {k: v.clone() for k, v in s["start"].items()}
        s["trace"] = L.new_trace(case["steps"], w, case["K"])
        s["params"] = L.BhParams(K=case["K"], kT=0.8, seed=seed, n_steps=case["steps"],
                                 min=_params(case))
        ctx.reserve(w * case["K"], n, s["params"].min.m)
        return s
    x, off = _displaced(case, seed)
    dev = x.device
    s["call"] = dict(n_cand=case["cand"])
    if off is None:
        s["call"].update(uniform_n=case["n"])
    else:
        s["call"].update(atom_offset=torch.as_tensor(off, device=dev), max_n=case["n"])
    s["energy"] = torch.empty(case["cand"], dtype=torch.float64, device=dev)
    if case["op"] == "eval":
        s["x"] = x.float() if case["prec"] == "f32" else x
        s["grad"] = torch.empty_like(s["x"])
        s["call"].update(prec=L.LJ_PREC_FP32 if case["prec"] == "f32" else L.LJ_PREC_FP64,
                         **_pot(case))
        return s
    s["x0"], s["x"] = x, torch.empty_like(x)
    s["status"] = torch.empty(case["cand"], dtype=torch.int32, device=dev)
    s["params"] = _params(case)
    if off is not None:
        # the first four atoms of each atom's cluster
        four = np.repeat(off[:-1], np.diff(off))[:, None] + np.arange(4)[None]
        s["four"] = torch.as_tensor(four, device=dev)
    ctx.reserve(case["cand"], case["n"], s["params"].m)
    return s


def _internal(x, four=None):
    """Distances of every atom to the first four of its cluster, FP32: (B, n, 3) -> (B, n, 4), or
    packed (total, 3) with their indices -> (total, 4)."""
    first = x[:, None, :4] if four is None else x[four]
    return torch.linalg.vector_norm((x[..., None, :] - first).float(), dim=-1)


def run(s):
    case, ctx = s["case"], s["ctx"]
    if case["op"] == "eval":
        L.lj_energy_grad_batched(ctx, s["x"], s["energy"], s["grad"], **s["call"])
        return dict(energy=s["energy"].float() if case["prec"] == "f32" else s["energy"],
                    grad=s["grad"])
    if case["op"] == "min":
        s["x"].copy_(s["x0"])
        L.lbfgs_minimize_batched(ctx, s["x"], s["energy"], s["status"], params=s["params"],
                                 **s["call"])
        shape = (case["cand"], case["n"], 3) if "four" not in s else (-1, 3)
        return dict(energy=s["energy"], status=s["status"],
                    distances=_internal(s["x"].view(shape), s.get("four")))
    for k, v in s["start"].items():
        s["state"][k].copy_(v)
    L.bh_step_batched(ctx, s["state"], s["params"], s["trace"])
    out = {k: v for k, v in s["state"].items() if not k.startswith("x_")}
    out.update({"trace_" + k: v for k, v in s["trace"].items() if k != "trial_iters"})
    for k in ("x_cur", "x_best"):
        out[k] = _internal(s["state"][k].view(case["walkers"], -1, 3))
    return out


# operations of one pair in one evaluation (fused multiply-adds counted twice, the reciprocal,
# square root and exponential once)
PAIR_FLOPS = dict(lj=28, morse=24)
# evaluations from displacements of this size to the stopping rule, a floor over what was seen
EVALS = 40


def work(case):
    sizes = _sizes(case) if case["op"] != "bh" else None
    if sizes is None:
        count = case.get("cand") or case["walkers"] * case["K"] * case["steps"]
        atoms, pairs = count * case["n"], count * case["n"] * (case["n"] - 1) / 2
    else:
        count, atoms = case["cand"], float(sizes.sum())
        pairs = float((sizes * (sizes - 1) / 2).sum())
    flops = PAIR_FLOPS[case["pot"]] * pairs
    if case["op"] == "eval":
        return dict(bytes=atoms * 6 * (4 if case["prec"] == "f32" else 8) + 8 * count,
                    flops=flops)
    if case["op"] == "min":
        return dict(bytes=atoms * 48 + 12 * count, flops=EVALS * flops)
    state = case["walkers"] * (case["n"] * 96 + 64) + 16 * count
    return dict(bytes=state, flops=EVALS * flops)


# ---------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------
def _pairs64(x, pot):
    """(B, n, 3) -> energies (B,) and gradients (B, n, 3)."""
    d = x[:, :, None] - x[:, None]
    r2 = d.square().sum(-1)
    r2.diagonal(dim1=1, dim2=2).fill_(1.0)
    if pot == "lj":
        s6 = r2 ** -3
        e, c = 4 * (s6 * s6 - s6), 24 * (s6 - 2 * s6 * s6) / r2
    else:
        r = r2.sqrt()
        m = torch.exp(MORSE_RHO * (1 - r))
        e, c = m * (m - 2), -2 * MORSE_RHO * m * (m - 1) / r
    e.diagonal(dim1=1, dim2=2).fill_(0.0)
    c.diagonal(dim1=1, dim2=2).fill_(0.0)
    return 0.5 * e.sum((1, 2)), (c[..., None] * d).sum(2)


def _hessian64(x, pot):
    n = x.shape[0]
    d = x[:, None] - x[None]
    r2 = d.square().sum(-1)
    r2.diagonal().fill_(1.0)
    if pot == "lj":                # a = V'(r) / r, b = (V''(r) - a) / r^2
        s6 = r2 ** -3
        a = 24 * (s6 - 2 * s6 * s6) / r2
        b = (672 * s6 * s6 - 192 * s6) / r2 ** 2
    else:
        r = r2.sqrt()
        m = torch.exp(MORSE_RHO * (1 - r))
        a = -2 * MORSE_RHO * m * (m - 1) / r
        b = (2 * MORSE_RHO ** 2 * m * (2 * m - 1) - a) / r2
    a.diagonal().fill_(0.0)
    b.diagonal().fill_(0.0)
    k = b[..., None, None] * d[..., :, None] * d[..., None, :] + \
        a[..., None, None] * torch.eye(3, dtype=x.dtype, device=x.device)
    h = -k
    i = torch.arange(n, device=x.device)
    h[i, i] = k.sum(1)
    return h.permute(0, 2, 1, 3).reshape(3 * n, 3 * n)


_RELAXED = {}


def _relaxed(n, pot):
    """The minimum of the structure of n atoms, (n, 3), and its energy: Newton steps with the
    rigid motions held and a shift that goes to zero.  Kept: it depends on n alone."""
    if (n, pot) not in _RELAXED:
        x = torch.as_tensor(_structure(n), device="cuda" if torch.cuda.is_available() else "cpu")
        eye = torch.eye(3 * n, dtype=x.dtype, device=x.device)
        for it in range(40):
            e, g = _pairs64(x[None], pot)
            c = x - x.mean(0)
            z = [torch.zeros_like(x) for _ in range(6)]
            for k in range(3):
                z[k][:, k] = 1.0
                z[3 + k][:, (k + 1) % 3] = -c[:, (k + 2) % 3]
                z[3 + k][:, (k + 2) % 3] = c[:, (k + 1) % 3]
            q = torch.linalg.qr(torch.stack([v.reshape(-1) for v in z], 1))[0]
            h = _hessian64(x, pot) + 100.0 * q @ q.T + (60.0 * 0.5 ** it if it < 24 else 0.0) * eye
            step = -torch.linalg.solve(h, g.reshape(-1))
            x = x + (step * min(1.0, 0.1 / float(step.abs().max()))).reshape(n, 3)
            if it > 24 and float(step.abs().max()) < 1e-13:
                break
        _RELAXED[n, pot] = (x, float(_pairs64(x[None], pot)[0]))
    return _RELAXED[n, pot]


def exact(case, seed):
    if case["op"] == "bh":
        w, t = case["walkers"], case["steps"]
        x, e = _relaxed(case["n"], case["pot"])
        d = _internal(x[None].repeat(w, 1, 1))
        e = torch.full((w,), e, dtype=torch.float64)
        return dict(e_cur=e, e_best=e, x_cur=d, x_best=d,
                    trace_trial_e=e[None, :, None].repeat(t, 1, case["K"]),
                    trace_best_trial_e=e[None].repeat(t, 1))
    if case["op"] == "min":
        sizes = _sizes(case)
        if case["n"] > ICO_MAX:    # a Hessian of thousands of rows, many times
            return None
        if sizes is None:
            x, e = _relaxed(case["n"], case["pot"])
            return dict(energy=torch.full((case["cand"],), e, dtype=torch.float64),
                        distances=_internal(x[None].repeat(case["cand"], 1, 1)))
        by_size = {int(k): _relaxed(int(k), case["pot"])[1] for k in np.unique(sizes)}
        return dict(energy=torch.tensor([by_size[int(k)] for k in sizes], dtype=torch.float64))
    x, off = _displaced(case, seed)
    if case["prec"] == "f32":
        x = x.float().double()
    x = x.view(-1, 3)
    if off is None:
        n = case["n"]
        xs = x.view(case["cand"], n, 3)
        got = [_pairs64(c, case["pot"]) for c in xs.split(max(1, 20_000_000 // (n * n)))]
        return dict(energy=torch.cat([e for e, _ in got]),
                    grad=torch.cat([g for _, g in got]).reshape(-1))
    sizes = np.diff(off)
    energy = torch.empty(case["cand"], dtype=torch.float64, device=x.device)
    grad = torch.empty_like(x)
    for n in np.unique(sizes):
        which = np.nonzero(sizes == n)[0]
        at = torch.as_tensor(off[which][:, None] + np.arange(n)[None], device=x.device)
        e, g = _pairs64(x[at], case["pot"])
        energy[torch.as_tensor(which, device=x.device)] = e
        grad[at.reshape(-1)] = g.reshape(-1, 3)
    return dict(energy=energy, grad=grad.reshape(-1))
