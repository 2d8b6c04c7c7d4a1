"""Several host threads at work on systems of their own: what one thread's
launches need must not depend on what another thread asks for."""
import threading

import numpy as np
import pytest

import synth
from test_gpu_track import ht  # noqa: F401  (the module's fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,large,small", [(1, 16, 6), (2, 28, 3), (4, 24, 3)])
def test_threads_tracking_systems_of_different_sizes(ht, L, large, small):  # noqa: F811
    """Two threads track systems of different sizes, whose kernels ask for
    different amounts of shared memory, at the same time on their own streams:
    every call succeeds with the bits of a run by itself."""
    m, calls = 40, 60

    def case(n):
        s = synth.total_degree_system(900 + n, n, 2 if n > 3 else 4, 6 if n < 4 else 10)
        out = dict(x=torch.zeros((n, 2, L, m), dtype=torch.float64, device="cuda"),
                   st=torch.zeros((m,), dtype=torch.int8, device="cuda"),
                   t=torch.zeros((m,), dtype=torch.float64, device="cuda"))
        # a call is mostly its launches: two steps a path, 64 captured rounds
        prm = ht.ht_default_params(L, max_steps=2, rounds_per_sync=64, iters_per_launch=1)
        return dict(sys=ht.system_from(s, L), deg=s.degrees(), out=out, prm=prm, stream=torch.cuda.Stream())

    def track(c):
        o = c["out"]
        ht.ht_track_paths(c["sys"], c["deg"], (0.6, 0.8), m, 0, None, c["prm"], o["x"], o["st"], o["t"], None, None,
                          c["stream"])

    cases = [case(large), case(small)]
    torch.cuda.synchronize()
    want = []
    for c in cases:
        track(c)
        torch.cuda.synchronize()
        want.append([v.cpu().numpy().copy() for v in c["out"].values()])
    errors = []
    start, done = threading.Barrier(2), threading.Event()

    def work(c, ref):  # the large system's calls, with the small one's until they end
        try:
            start.wait()
            k = 0
            while k < calls if c is cases[0] else not done.is_set():
                k += 1
                track(c)
                c["stream"].synchronize()
                if not all(np.array_equal(v.cpu().numpy(), r, equal_nan=True) for v, r in zip(c["out"].values(), ref)):
                    raise AssertionError("the results differ from a run by itself")
        except Exception as e:  # noqa: BLE001  (reported by the main thread)
            errors.append(repr(e))
        finally:
            done.set()

    threads = [threading.Thread(target=work, args=cr) for cr in zip(cases, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
