"""The tracker's tuner against the automatic launch shape, and the cache's key."""
import json
import time

import numpy as np
import pytest

import synth
from paper_1505_00383_gb300 import ht, tuning


def test_cache_key_changes_with_the_kernels(tmp_path, monkeypatch):
    """A shape tuned on other kernels is not reused."""
    path = str(tmp_path / "tune.json")
    s = synth.config_system("plain_n6_d")
    calls = []

    def fake(handle, deg, gamma, n, params):
        calls.append(n)
        return 4, 2, 1.0

    p = ht.ht_params()
    for version in ("a", "b", "b"):
        monkeypatch.setattr(tuning, "kernels_id", lambda v=version: v)
        tuning.tuned_track_shape("H", s, 1, (1.0, 0.0), 64, p, path, "G", tune=fake)
    assert len(calls) == 2 and len(json.load(open(path))) == 2


def test_kernels_id_is_of_the_sources():
    assert len(tuning.kernels_id()) == 12 and tuning.kernels_id() == tuning.kernels_id()


@pytest.mark.gpu
@pytest.mark.parametrize("L,n", [(2, 5), (4, 5), (2, 3)])
def test_tuning_is_no_slower_than_not_tuning(L, n):
    """DD and QD systems of few variables, whose automatic teams are wider than
    any fixed one up to n: a tuned system tracks as fast as an untuned one
    (fixed teams of at most four warps took 1.25 times as long; the best of
    five runs of each, 1.12 for what runs differ by) and to the same bits."""
    torch = pytest.importorskip("torch")
    from paper_1505_00383_gb300 import _build
    _build.build()
    s = synth.total_degree_system(900 + n, n, 2, 6)
    m = 2 ** n
    prm = ht.ht_default_params(L, h_min=1e-6, max_steps=60)
    x = torch.zeros((n, 2, L, m), dtype=torch.float64, device="cuda")
    st = torch.zeros((m,), dtype=torch.int8, device="cuda")
    t = torch.zeros((m,), dtype=torch.float64, device="cuda")
    plain, tuned = ht.system_from(s, L), ht.system_from(s, L)
    team, iters, _ = ht.ht_tune_track(tuned, s.degrees(), (0.6, 0.8), m, prm)
    assert team in (0, 1, 2, 4, 8) and iters in (2, 4, 8)
    best, ends = {}, {}
    for _ in range(5):
        for name, hs in (("plain", plain), ("tuned", tuned)):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            ht.ht_track_paths(hs, s.degrees(), (0.6, 0.8), m, 0, None, prm, x, st, t)
            torch.cuda.synchronize()
            best[name] = min(best.get(name, 1e9), time.perf_counter() - t0)
            ends[name] = (x.cpu().numpy(), st.cpu().numpy())
    assert best["tuned"] <= 1.12 * best["plain"], best
    assert all(np.array_equal(a, b, equal_nan=True) for a, b in zip(ends["plain"], ends["tuned"]))
