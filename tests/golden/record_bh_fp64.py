"""FP64 Basin Hopping traces for bh_fp64_traces.json: how every trial ended and the bits of its
energy.

At the default gtol the last line search of an FP64 minimisation has to resolve decreases below an
ulp of the energy, so the status of a trial records the order and the rounding of every sum that
led to it.  The stored traces are those of pairs in row-major order of the upper triangle (one-sided
rows above 64 atoms), correctly rounded reciprocals and the recursion's products summed atom by
atom.  They change only with a deliberate change of that arithmetic, and are then recorded
again on a GPU:  python tests/golden/record_bh_fp64.py
"""
import json
import os
import sys

import numpy as np
import torch

HERE = os.path.dirname(os.path.abspath(__file__))
PATH = os.path.join(HERE, "bh_fp64_traces.json")

# teams of one and two warps, one and two atoms a thread, with and without a pair buffer
CASES = {
    "lj13": dict(n=13, walkers=4, K=1, steps=50, step=0.15, pot="lj"),
    "lj38": dict(n=38, walkers=2, K=4, steps=8, step=0.15, pot="lj"),
    "lj55": dict(n=55, walkers=1, K=4, steps=6, step=0.08, pot="lj", team=32),
    "lj77": dict(n=77, walkers=2, K=4, steps=5, step=0.08, pot="lj"),
    "lj140": dict(n=140, walkers=1, K=4, steps=2, step=0.08, pot="lj"),
    "morse13": dict(n=13, walkers=2, K=2, steps=10, step=0.15, pot="morse"),
    "morse77": dict(n=77, walkers=1, K=4, steps=2, step=0.08, pot="morse"),
}


def start(n):
    """(n, 3) sites that every machine computes alike: an icosahedron of 13, else the first n
    sites of an fcc lattice by distance."""
    if n == 13:
        s = [(0.0, 0.0, 0.0)]
        for a in (0.57, -0.57):
            for b in (0.9223, -0.9223):
                s += [(0.0, a, b), (a, b, 0.0), (b, 0.0, a)]
        return np.array(s)
    r = range(-6, 7)
    p = sorted((x * x + y * y + z * z, x, y, z) for x in r for y in r for z in r
               if (x + y + z) % 2 == 0)
    return np.array([q[1:] for q in p[:n]], dtype=np.float64) * 0.79


def run(lj, c):
    n, w = c["n"], c["walkers"]
    x = torch.as_tensor(np.tile(start(n).reshape(1, -1), (w, 1)), device="cuda")
    f = dict(device="cuda", dtype=torch.float64)
    state = dict(x_cur=x, e_cur=torch.zeros(w, **f), x_best=x.clone(), e_best=torch.zeros(w, **f),
                 stepsize=torch.full((w,), c["step"], **f),
                 win_accept=torch.zeros(w, dtype=torch.int32, device="cuda"),
                 n_accept=torch.zeros(w, dtype=torch.int32, device="cuda"))
    trace = lj.new_trace(c["steps"], w, c["K"])
    pot = lj.LJ_POT_MORSE if c["pot"] == "morse" else lj.LJ_POT_LJ
    params = lj.BhParams(K=c["K"], kT=0.8, seed=11, n_steps=c["steps"],
                         min=lj.LbfgsParams(prec=lj.LJ_PREC_FP64, potential=pot, rho=6.0))
    ctx = lj.Ctx(0)
    if "team" in c:
        ctx.set_option(lj.LJ_OPT_BH_TEAM, c["team"])
    lj.bh_step_batched(ctx, state, params, trace)
    torch.cuda.synchronize()
    ctx.close()
    return dict(status="".join(str(v) for v in trace["trial_status"].cpu().reshape(-1).tolist()),
                energy=[v.hex() for v in trace["trial_e"].cpu().reshape(-1).tolist()])


def main():
    sys.path.insert(0, os.path.dirname(os.path.dirname(HERE)))
    from paper_2510_25938_gb300 import lj_bh
    with open(PATH, "w") as f:
        json.dump({k: run(lj_bh, c) for k, c in CASES.items()}, f, indent=0)
        f.write("\n")


if __name__ == "__main__":
    main()
