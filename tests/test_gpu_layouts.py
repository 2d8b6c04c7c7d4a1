"""The double tracker's least squares in its three layouts -- a column per lane
(few paths), a system per lane in the wide kernel (up to one group of 32 an SM)
and in the 8-warp kernel (more) -- and for every team size.  All perform the
same operations in the same order, so no layout may show in a result.  The
numbers of paths come from the SM count, so that each run takes the layout that
it names whatever the chip."""
import numpy as np
import pytest

import synth
from test_gpu_track import ht, track_gpu  # noqa: F401  (ht: the module's fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _column_paths(n, nrhs):
    """Paths up to which the tracker solves with a column per lane."""
    return torch.cuda.get_device_properties(0).multi_processor_count * 4 * (32 // (n + nrhs - 1)) if n <= 16 else 0


def _run(ht, s, m, first=0, **over):  # noqa: F811
    out = track_gpu(ht, s, 1, m, first=first, h_min=1e-4, **over)
    return [np.asarray(out[k]) for k in ("x_end", "status", "t_end", "steps")]


@pytest.mark.parametrize("nrhs", [1, 2])
@pytest.mark.parametrize("n", list(range(2, 17)))
def test_columns_per_lane_match_systems_per_lane(ht, n, nrhs):  # noqa: F811
    """n = 2 to 16 (every unrolled body of the column layout, at and below its
    size): the first paths of a run too large for the column layout, tracked
    by a system per lane until few are left, and by themselves in the column
    layout from the first round.  Six steps a path, so that the large run's
    paths are all still active when its layout is chosen."""
    limit = _column_paths(n, nrhs)
    many, few = limit + 33, min(limit, 37)
    s = synth.total_degree_system(700 + n, n, 2 if n > 3 else 5, 6 if n == 2 else 8)
    over = dict(predictor=2 if nrhs == 2 else 0, max_steps=6, iters_per_launch=1, rounds_per_sync=2)
    whole = _run(ht, s, many, **over)
    part = _run(ht, s, few, **over)
    for a, b in zip(whole, part):
        assert np.array_equal(a[..., :few], b, equal_nan=True)
    part = _run(ht, s, few, first=many - few, **over)
    for a, b in zip(whole, part):
        assert np.array_equal(a[..., -few:], b, equal_nan=True)
    assert np.min(whole[3]) >= 1


@pytest.mark.parametrize("n,predictor", [(6, 0), (6, 2), (16, 0), (16, 2), (19, 0)])
def test_team_sizes_with_a_system_per_lane(ht, n, predictor):  # noqa: F811
    """Teams of 1 to 16 warps where a system stays on its lane: in the wide
    kernel (at most a group an SM), the same bits as the automatic choice, and
    in the 8-warp kernel (more groups than SMs)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    limit = _column_paths(n, 2 if predictor else 1)
    s = synth.total_degree_system(720 + n, n, 2, 8)
    for m, teams in ((limit + 5, (1, 2, 4, 8, 16)), (32 * sms + 7, (1, 4, 8))):
        assert m > limit
        over = dict(predictor=predictor, max_steps=4, iters_per_launch=1, rounds_per_sync=2)
        base = _run(ht, s, m, **over)
        for tw in teams:
            for a, b in zip(base, _run(ht, s, m, team_warps=tw, **over)):
                assert np.array_equal(a, b, equal_nan=True), (m, tw)


@pytest.mark.parametrize("predictor", [0, 2])
@pytest.mark.parametrize("L,n", [(2, 1), (2, 2), (2, 3), (2, 5), (2, 17), (4, 1), (4, 2), (4, 3), (4, 9), (4, 17)])
def test_integer_groups_of_more_paths_than_sms_hold(ht, L, n, predictor):  # noqa: F811
    """DD and QD with more groups than SMs: teams of the warps that have work,
    32 to 1 systems a warp in the solve, groups of equal size where a warp
    takes one; against few paths (the widest teams, columns over slots)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    s = synth.total_degree_system(740 + n, n, 2 if n > 3 else 5, 6 if n > 1 else 4)
    over = dict(h_min=1e-4, predictor=predictor, max_steps=4, iters_per_launch=1, rounds_per_sync=2)
    many, few = 32 * sms + 77, 41
    keys = ("x_end", "status", "t_end", "steps")
    whole = track_gpu(ht, s, L, many, **over)
    for first in (0, many - few):
        part = track_gpu(ht, s, L, few, first=first, **over)
        for k in keys:
            assert np.array_equal(np.asarray(whole[k])[..., first:first + few], np.asarray(part[k]), equal_nan=True), k


def test_integer_workspace_follows_the_number_of_paths(ht):  # noqa: F811
    """QD, n = 24, one path an SM: the matrices of those paths (48 KB each) and
    not of 32 paths a CTA (1.5 MB each, 233 MB on 152 SMs); 48 KB and its state of
    about 5 KB a path stay below 128 KB a path."""
    m = torch.cuda.get_device_properties(0).multi_processor_count
    s = synth.total_degree_system(760, 24, 2, 6)
    hs = ht.system_from(s, 4)
    x = torch.zeros((24, 2, 4, m), dtype=torch.float64, device="cuda")
    st = torch.zeros((m,), dtype=torch.int8, device="cuda")
    t = torch.zeros((m,), dtype=torch.float64, device="cuda")
    prm = ht.ht_default_params(4, max_steps=1)
    # the kernels' local memory is allocated on their first launch
    warm = ht.system_from(s, 4)
    ht.ht_track_paths(warm, s.degrees(), (0.6, 0.8), m, 0, None, prm, x, st, t)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ht.ht_track_paths(hs, s.degrees(), (0.6, 0.8), m, 0, None, prm, x, st, t)
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= m * (128 << 10) + (4 << 20)
