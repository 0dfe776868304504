"""Cases of the KIN_DEBUG build at the launch shapes that the library chooses
itself: LBE steps in pairs, DUGKS tiles of 5, 8 and 11 rows (FP64 3 and 7), whole
rows in a warp, the velocity written by the step, statistics, and ensembles.

Run by tests/test_gpu_debug_shapes.py in a process of its own (a process loads
one build of the library).  Prints one JSON line: per case the error against the
FP64 oracle, that of E, the debug status and the guard check.
"""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

import kin_inputs as ki  # noqa: E402
import oracle  # noqa: E402
import paper_1601_03815_gb300 as kin  # noqa: E402

NU = 0.013
F32, F16, BF16, F64 = kin.F32, kin.F16, kin.BF16, kin.F64
# (scheme, storage, N, steps)
CASES = [("lbe", F32, N, n) for N, n in ((2, 2), (5, 3), (31, 2), (32, 3), (48, 2), (89, 3), (97, 2))]
CASES += [("lbe", F16, N, 3) for N in (2, 5, 12, 32, 34)] + [("lbe", BF16, 9, 2), ("lbe", F64, 33, 2)]
CASES += [("dugks", F32, N, 2) for N in (3, 12, 30, 31, 32, 33, 45, 64, 97)]
CASES += [("dugks", F64, N, 1) for N in (5, 31, 32, 33, 45)] + [("dugks", F16, N, 2) for N in (12, 33, 38)]


def state(N, seed):
    u = ki.random_velocity(N, N, N, seed, 0.03)
    return oracle.equilibrium_field(u) + ki.random_populations(N, N, N, seed + 1, 2e-5)


def make(scheme, storage, N, seed):
    sim = kin.Sim(N, kin.LBE_MRT if scheme == "lbe" else kin.DUGKS, NU, 0.1, 1.0 if scheme == "lbe" else 0.5, storage)
    sim.set_f(state(N, seed))
    return sim


def stepped(scheme, f, n):
    for _ in range(n):
        f = oracle.step(scheme, f, NU, 1.0 if scheme == "lbe" else 0.5)
    return f


def err(got, ref):
    scale = np.abs(ref).reshape(19, -1).max(axis=1)
    return float((np.abs(got - ref).reshape(19, -1).max(axis=1) / scale).max())


def status(sims):
    guards = "ok"
    for sim in sims:
        try:
            sim.check_guards()
        except kin.KinError as exc:
            guards = str(exc)
    return {"debug_word": kin.debug_status(reset=True)[1], "guards": guards}


def main():
    kin.load(debug=True)
    oracle.build()
    out = {"debug_build": kin.debug_status()[0], "cases": []}
    for scheme, storage, N, n in CASES:
        sim = make(scheme, storage, N, 60 + N)
        f_in = sim.get_f()
        # n steps, of which the last also makes the statistics
        E = sim.step_stats(n)[0]
        got = sim.get_f()
        Eo = oracle.stats(got, NU)[0]
        out["cases"].append({"scheme": scheme, "storage": storage, "N": N, "steps": n,
                             "err": err(got, stepped(scheme, f_in, n)), "err_E": abs(E / Eo - 1), **status([sim])})
        sim.close()
    for specs in ([("dugks", F32, 12), ("dugks", F32, 33), ("lbe", F32, 9)],
                  [("dugks", F16, 12), ("dugks", F16, 34), ("lbe", F16, 8)],
                  [("dugks", F32, 33), ("dugks", F16, 16), ("dugks", BF16, 10), ("lbe", BF16, 10), ("lbe", F32, 5)]):
        sims = [make(scheme, storage, N, 80 + k) for k, (scheme, storage, N) in enumerate(specs)]
        states = [s.get_f() for s in sims]
        ens = kin.Ensemble(sims)
        ens.step(2)
        for sim, f, (scheme, storage, N) in zip(sims, states, specs):
            got = sim.get_f()
            E, Eo = sim.stats()[0], oracle.stats(got, NU)[0]
            out["cases"].append({"scheme": "ensemble " + scheme, "storage": storage, "N": N, "steps": 2,
                                 "err": err(got, stepped(scheme, f, 2)), "err_E": abs(E / Eo - 1), **status(sims)})
        ens.close()
        for sim in sims:
            sim.close()
    print(json.dumps(out))


if __name__ == "__main__":
    main()
