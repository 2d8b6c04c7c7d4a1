"""The rule that deals a polynomial's monomials to several warps, against
measured times (CPU: the rule is host code).

golden/eval_split_us.json holds microseconds of ht_eval_diff, variant 2 with
256 threads, on a GB300 of 152 SMs: with S = 1, 2, 3, 4, 5, 8 and 16 warps a
polynomial, and of the kernel that preceded splitting (one warp always)."""
import ctypes
import json
import os
import subprocess

import numpy as np
import pytest

import synth

HERE = os.path.dirname(os.path.abspath(__file__))
SIZES = (1, 2, 3, 4, 5, 8, 16)


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("split") / "libsplit_shim.so")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-o", out, os.path.join(HERE, "split_shim.cpp")])
    lib = ctypes.CDLL(out)
    lib.split_steps.restype = ctypes.c_int64
    lib.split_steps.argtypes = [ctypes.c_void_p, ctypes.c_int]
    lib.split_pick.argtypes = [ctypes.c_int] * 3 + [ctypes.c_int64, ctypes.c_double, ctypes.c_int, ctypes.c_int64,
                                                    ctypes.c_int64]
    return lib


def _shape(lib, s):
    steps, row = [], 0
    for t in s.n_terms:
        n = 0
        for e in s.exps[row:row + t]:
            v = np.flatnonzero(e)
            pr = np.ascontiguousarray(v | (e[v].astype(np.int64) << 8), dtype=np.uint16)
            n += lib.split_steps(pr.ctypes.data, len(v))
        steps.append(n)
        row += t
    return s.n_vars, s.n_polys, int(max(s.n_terms)), max(steps), float(np.mean(steps))


def test_picks_are_near_the_best_measured_split(shim):
    """Where the pick was measured: at most 1.25 times the best S (the model's
    constants leave 1.21), and never more than one warp a polynomial took."""
    rows = json.load(open(os.path.join(HERE, "golden", "eval_split_us.json")))["rows"]
    shapes, ratios = {}, []
    for name, limbs, n, unsplit, *us in rows:
        if name not in shapes:
            shapes[name] = _shape(shim, synth.config_system(name))
        pick = shim.split_pick(*shapes[name], limbs, (n + 31) // 32, 152)
        S, G = divmod(pick, 100)
        assert 1 <= S <= shapes[name][2] and 1 <= G <= shapes[name][1] and (S == 1 or S * G <= 16)
        if S not in SIZES:
            continue
        t, best = us[SIZES.index(S)], min(u for k, u in zip(SIZES, us) if k <= shapes[name][2])
        assert t <= 1.25 * best and t <= unsplit, (name, limbs, n, S, t, best, unsplit)
        ratios.append(t / best)
    assert len(ratios) > 0.7 * len(rows) and np.exp(np.mean(np.log(ratios))) < 1.03


@pytest.mark.parametrize("limbs", [1, 2, 4])
def test_every_shape_gets_a_valid_split(shim, limbs):
    """Extremes of the rule's domain: one term, one polynomial, many of either."""
    for nv in (1, 7, 64):
        for np_ in (1, 5, 33, 1000):
            for terms in (1, 2, 17, 5000):
                for blocks in (1, 3, 152, 100000):
                    S, G = divmod(shim.split_pick(nv, np_, terms, terms * 3, terms * 2.5, limbs, blocks, 152), 100)
                    assert 1 <= S <= min(16, terms) and 1 <= G <= np_
                    assert S * G <= (16 if S > 1 or limbs == 4 else 32)
