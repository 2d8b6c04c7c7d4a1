"""What the library is measured on: its public calls at the sizes of its own workloads.

Five kinds of call, each through the ctypes binding as a program calls it:

* ``eval``    ht_eval_diff: every polynomial and the Jacobian at a batch of points, in double (the default
              kernel choice) and in double double and quad double (the integer-limb kernel that the
              autotuner keeps for them, set here by name so that both sides of a comparison run it);
* ``track``   ht_track_paths_ex: whole paths of the total-degree homotopy, with the plain step rule or the
              network's proposals, by extrapolation or on tangents;
* ``refine``  ht_track_refined: tracking in double, refinement of every endpoint in more limbs;
* ``mgs``     ht_mgs_solve_ex: batched least squares, the corrector's linear solve by itself;
* ``mlp``     ht_mlp_train: training the step-size network.

The supports of the polynomial systems are the ones of the synthetic workloads; coefficients, points,
gamma, matrices and samples come from the case's seed.
"""
import functools
import math

import numpy as np
import torch

import synth
from paper_1505_00383_gb300 import ht, learned

# Newton rounds per path of the tracking workloads (step floor 1e-9), for the work estimates
ROUNDS = {"plain_n6_d": 300, "learned_n16_d": 410, "batched_n12_dd": 330, "stress_n10_qd": 357}
TRACK = {"plain_n6_d": (1, 64), "learned_n16_d": (1, 16384), "batched_n12_dd": (2, 4096), "stress_n10_qd": (4, 4096)}
EVAL_MAX = {"evaldiff_n32": 65536, "cyclic10_shape": 65536, "nash8_shape": 32768, "pieri44_shape": 8192,
            "batched_n12_dd": 65536, "stress_n10_qd": 65536}


def listed():
    return [
        # the smallest batch of the paper's evaluation tables: latency and launches
        dict(name="eval_d_small", kind="eval", system="cyclic10_shape", limbs=1, points=10),
        # the evaluation sweep of the benchmark, one call per precision
        dict(name="eval_d", kind="eval", system="evaldiff_n32", limbs=1, points=65536),
        dict(name="eval_dd", kind="eval", system="evaldiff_n32", limbs=2, points=65536),
        dict(name="eval_qd", kind="eval", system="evaldiff_n32", limbs=4, points=65536),
        # an ordinary batch of the paper's tables that does not fill the last block of points
        dict(name="eval_qd_ragged", kind="eval", system="pieri44_shape", limbs=4, points=999),
        # all 64 paths of the smallest workload: latency of whole runs
        dict(name="track_d_small", kind="track", system="plain_n6_d", paths=64, predictor=0, net=False),
        # a quarter of the n = 16 workload in double: several groups of paths per SM and a long tail
        dict(name="track_d", kind="track", system="learned_n16_d", paths=16384, predictor=0, net=False),
        # every path of the batched double double workload: fewer groups of paths than SMs
        dict(name="track_dd", kind="track", system="batched_n12_dd", paths=4096, predictor=0, net=False),
        # part of the quad double stress workload, with its faster predictor (cubic Hermite on tangents)
        dict(name="track_qd", kind="track", system="stress_n10_qd", paths=4096, predictor=2, net=False),
        # "quality up": double tracking, double double endpoints
        dict(name="refine_dd", kind="refine", system="batched_n12_dd", limbs=2, paths=4096),
        # the corrector's solve by itself, at the quad double workload's shape
        dict(name="mgs_qd", kind="mgs", limbs=4, variant=2, rows=10, cols=10, systems=16384),
        # training of the step-size network, four passes over recorded steps
        dict(name="mlp_train", kind="mlp", samples=50000, batch=4096, epochs=4),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "track", "track", "refine", "mgs", "mlp"])
    if kind == "eval":
        system = rng.choice(sorted(EVAL_MAX))
        return dict(kind=kind, system=system, limbs=rng.choice([1, 2, 4]), points=_log(rng, 10, EVAL_MAX[system]))
    if kind == "track":
        system = rng.choice(sorted(TRACK))
        limbs, most = TRACK[system]
        return dict(kind=kind, system=system, paths=_log(rng, 16, most // 2),
                    predictor=2 if limbs == 4 else rng.choice([0, 0, 2]), net=limbs == 1 and rng.random() < 0.4)
    if kind == "refine":
        return dict(kind=kind, system="batched_n12_dd", limbs=2, paths=_log(rng, 32, 4096))
    if kind == "mgs":
        limbs = rng.choice([1, 2, 4])
        cols = rng.randint(2, 16)
        return dict(kind=kind, limbs=limbs, variant=0 if limbs == 1 else rng.choice([0, 2]), rows=cols + rng.choice([0, 0, 1, 3]),
                    cols=cols, systems=_log(rng, 30, 65536 // (limbs * limbs)))
    return dict(kind=kind, samples=_log(rng, 500, 50000), batch=rng.choice([512, 1000, 4096]), epochs=rng.randint(1, 4))


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=None)
def _support(name):
    return synth.config_system(name)


def _system(name, seed):
    """The workload's supports with coefficients on the unit circle drawn from the seed."""
    s = _support(name)
    th = np.random.RandomState(seed % (1 << 31)).uniform(0.0, 2.0 * np.pi, s.n_monomials)
    return synth.System(n_vars=s.n_vars, n_polys=s.n_polys, n_terms=s.n_terms, exps=s.exps,
                        coef=np.ascontiguousarray(np.stack([np.cos(th), np.sin(th)], axis=1)))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _limbs(lead, limbs, g):
    """lead (any shape) as limbs non-overlapping doubles: [limbs] + shape."""
    out = [lead]
    for _ in range(1, limbs):
        ulp = torch.abs(torch.nextafter(out[-1], torch.full_like(lead, math.inf)) - out[-1])
        out.append(ulp * (torch.rand(lead.shape, dtype=torch.float64, device="cuda", generator=g) - 0.5))
    return torch.stack(out)


def _points(n_vars, n_pts, limbs, seed):
    """Points with |x_i| = 1: [n_vars][2][limbs][n_pts]."""
    g = _gen(seed)
    th = 2.0 * math.pi * torch.rand((n_vars, n_pts), dtype=torch.float64, device="cuda", generator=g)
    x = torch.stack([_limbs(torch.cos(th), limbs, g), _limbs(torch.sin(th), limbs, g)])  # [2][L][nv][n]
    return x.permute(2, 0, 1, 3).contiguous()


def _matrices(case, seed):
    """Augmented matrices [A | b]: [rows][cols + 1][2][limbs][systems], entries in the unit square."""
    g = _gen(seed)
    shape = (2, case["rows"], case["cols"] + 1, case["systems"])
    a = _limbs(2.0 * torch.rand(shape, dtype=torch.float64, device="cuda", generator=g) - 1.0, case["limbs"], g)
    return a.permute(2, 3, 1, 0, 4).contiguous()


def _outputs(n, limbs, m):
    return dict(x=torch.empty((n, 2, limbs, m), dtype=torch.float64, device="cuda"),
                status=torch.empty((m,), dtype=torch.int8, device="cuda"),
                t=torch.empty((m,), dtype=torch.float64, device="cuda"),
                steps=torch.empty((m,), dtype=torch.int32, device="cuda"))


def _samples(n, seed):
    """Features as the tracker computes them (t, logarithms of steps and norms, flags) and step labels."""
    g = _gen(seed)
    x = 2.0 * torch.rand((n, ht.HT_MLP_IN), device="cuda", generator=g) - 1.0
    x[:, 11:] = 0.0
    y = torch.stack([0.5 * x[:, 1] - 0.3 * x[:, 3] + 0.2 * torch.sin(3.0 * x[:, 2]), 0.1 * x[:, 9]], dim=1)
    return x.contiguous(), (y + 0.05 * torch.randn(y.shape, device="cuda", generator=g)).contiguous()


def prepare(case, seed):
    kind, st = case["kind"], {"case": case}
    if kind == "eval":
        s, L, n = _system(case["system"], seed), case["limbs"], case["points"]
        st["sys"] = ht.system_from(s, L)
        if L > 1:
            ht.ht_set_eval_config(st["sys"], 2, 256)
        st["x"] = _points(s.n_vars, n, L, seed)
        st["val"] = torch.empty((s.n_polys, 2, L, n), dtype=torch.float64, device="cuda")
        st["jac"] = torch.empty((s.n_polys, s.n_vars, 2, L, n), dtype=torch.float64, device="cuda")
    elif kind in ("track", "refine"):
        s, m = _system(case["system"], seed), case["paths"]
        L = TRACK[case["system"]][0] if kind == "track" else case["limbs"]
        st["deg"] = s.degrees()
        st["gamma"] = synth.random_gamma(seed)
        st["sys"] = ht.system_from(s, L)
        st["params"] = ht.ht_default_params(L, h_min=1e-9, predictor=case.get("predictor", 0))
        st["out"] = _outputs(s.n_vars, L, m)
        if kind == "refine":
            st["lo"] = ht.system_from(s, 1)
            st["params_lo"] = ht.ht_default_params(1, h_min=1e-9)
        if case.get("net"):
            st["net"] = ht.ht_mlp_create()
            ht.ht_mlp_set_params(st["net"], learned.init_params(seed))
            st["io"] = ht.ht_track_io(mlp=st["net"].handle, fallback_steps=1, rho_min=learned.RHO_RANGE[0],
                                      rho_max=learned.RHO_RANGE[1])
    elif kind == "mgs":
        L, cols = case["limbs"], case["cols"]
        st["a"] = _matrices(case, seed)
        st["work"] = torch.empty_like(st["a"])
        st["r"] = torch.zeros((cols, cols + 1, 2, L, case["systems"]), dtype=torch.float64, device="cuda")
        st["x"] = torch.empty((cols, 2, L, case["systems"]), dtype=torch.float64, device="cuda")
    else:
        st["x"], st["y"] = _samples(case["samples"], seed)
        st["p0"] = learned.init_params(seed)
        st["net"] = ht.ht_mlp_create()
    return st


# --------------------------------------------------------------------- run
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "eval":
        ht.ht_eval_diff(state["sys"], case["points"], state["x"], state["val"], state["jac"])
        return {"val": state["val"], "jac": state["jac"]}
    if kind == "track":
        o = state["out"]
        ht.ht_track_paths_ex(state["sys"], state["deg"], state["gamma"], case["paths"], 0, None, state["params"],
                             o["x"], o["status"], o["t"], o["steps"], None, state.get("io"))
        return o
    if kind == "refine":
        o = state["out"]
        ht.ht_track_refined(state["lo"], state["sys"], state["deg"], state["gamma"], case["paths"], 0,
                            state["params_lo"], state["params"], o["x"], o["status"], o["t"])
        return {k: o[k] for k in ("x", "status", "t")}
    if kind == "mgs":
        state["work"].copy_(state["a"])  # the solve overwrites its matrix
        ht.ht_mgs_solve_ex(case["limbs"], case["variant"], case["rows"], case["cols"], case["systems"],
                           state["work"], state["r"], state["x"])
        return {"q": state["work"], "r": state["r"], "x": state["x"]}
    ht.ht_mlp_set_params(state["net"], state["p0"])
    losses = ht.ht_mlp_train(state["net"], case["samples"], state["x"], state["y"], case["epochs"], case["batch"], 2e-3)
    return {"losses": losses, "params": ht.ht_mlp_get_params(state["net"])}


# -------------------------------------------------------------------- work
def _eval_flops(name):
    """Flops of one evaluation of values and Jacobian (complex multiply 6, add 2)."""
    e = _support(name).exps.astype(int)
    k, extra = (e > 0).sum(axis=1), np.maximum(e - 1, 0).sum(axis=1)
    muls = np.where(k == 0, 0, extra + np.where(k == 1, 1, 3 * k - 3))
    return float((6 * muls + 2 * (k + 1)).sum())


def work(case):
    kind = case["kind"]
    if kind == "eval":
        s, L, n = _support(case["system"]), case["limbs"], case["points"]
        return {"bytes": 16.0 * L * n * (s.n_vars + s.n_polys * (s.n_vars + 1)),
                "flops": _eval_flops(case["system"]) * n}
    if kind in ("track", "refine"):
        n, m = _support(case["system"]).n_vars, case["paths"]
        L = TRACK[case["system"]][0] if kind == "track" else case["limbs"]
        rounds = ROUNDS[case["system"]] * m  # each: an evaluation and a least-squares solve
        return {"bytes": 16.0 * L * n * m + 13.0 * m, "flops": rounds * (_eval_flops(case["system"]) + 8.0 * n ** 3)}
    if kind == "mgs":
        r, c, m = case["rows"], case["cols"], case["systems"]
        return {"bytes": 16.0 * case["limbs"] * m * (2.0 * r * (c + 1) + c * (c + 1) / 2 + 2 * c),
                "flops": 8.0 * m * (r * c * (c + 1) + c * c / 2)}
    n = float(case["samples"]) * case["epochs"]
    return {"bytes": n * 4 * (ht.HT_MLP_IN + ht.HT_MLP_OUT), "flops": 6.0 * n * ht.HT_MLP_NPARAM}


# ------------------------------------------------------------------- exact
def exact(case, seed):
    """Values from complex doubles; in more limbs the leading limb carries the value and the others are zero."""
    if case["kind"] == "eval":
        return _exact_eval(case, seed)
    if case["kind"] == "mgs":
        a = _matrices(case, seed)[:, :, :, 0]
        z = torch.complex(a[:, :, 0], a[:, :, 1]).permute(2, 0, 1)  # [systems][rows][cols + 1]
        q, r = torch.linalg.qr(z[:, :, :-1])
        x = torch.linalg.solve_triangular(r, q.mH @ z[:, :, -1:], upper=True)[:, :, 0].T  # [cols][systems]
        out = torch.zeros((case["cols"], 2, case["limbs"], case["systems"]), dtype=torch.float64, device="cuda")
        out[:, 0, 0], out[:, 1, 0] = x.real, x.imag
        return {"q": None, "r": None, "x": out}
    return None


def _exact_eval(case, seed):
    s, L, n = _system(case["system"], seed), case["limbs"], case["points"]
    p = _points(s.n_vars, n, L, seed)[:, :, 0]
    x = torch.complex(p[:, 0], p[:, 1])
    val = torch.zeros((s.n_polys, 2, L, n), dtype=torch.float64, device="cuda")
    jac = torch.zeros((s.n_polys, s.n_vars, 2, L, n), dtype=torch.float64, device="cuda")
    top = int(s.exps.max())
    pw = [torch.ones_like(x)]
    for _ in range(top):
        pw.append(pw[-1] * x)
    row = 0
    for j in range(s.n_polys):
        v = torch.zeros((n,), dtype=torch.complex128, device="cuda")
        d = torch.zeros((s.n_vars, n), dtype=torch.complex128, device="cuda")
        for _ in range(int(s.n_terms[j])):
            c = complex(s.coef[row, 0], s.coef[row, 1])
            sup = [(i, int(s.exps[row, i])) for i in np.flatnonzero(s.exps[row])]
            row += 1
            pre = [torch.full_like(v, c)]
            for i, a in sup:
                pre.append(pre[-1] * pw[a][i])
            v += pre[-1]
            suf = None
            for r in range(len(sup) - 1, -1, -1):
                i, a = sup[r]
                t = pre[r] * (pw[a - 1][i] * a)
                d[i] += t if suf is None else t * suf
                suf = pw[a][i] if suf is None else suf * pw[a][i]
        val[j, 0, 0], val[j, 1, 0] = v.real, v.imag
        jac[j, :, 0, 0], jac[j, :, 1, 0] = d.real, d.imag
    return {"val": val, "jac": jac}
