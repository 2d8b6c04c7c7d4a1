"""The layouts that the least squares and the tracker choose by size: one
matrix row per lane (DD, QD), one column per lane (double, few paths), columns
of a system over several slots, groups of fewer than 32 paths.  None of them
may show in a result."""
import numpy as np
import pytest

import synth
from test_gpu_track import _mgs_case, ht, track_gpu  # noqa: F401  (ht: the module's fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [2, 4])
@pytest.mark.parametrize("rows,cols", [(1, 1), (2, 1), (3, 3), (4, 4), (5, 2), (8, 8), (9, 9), (11, 10), (16, 16), (17, 5),
                                       (31, 30), (32, 32), (33, 33)])
def test_integer_least_squares_at_the_edges_of_the_row_layout(ht, L, rows, cols):  # noqa: F811
    """8, 4, 3, 2 and 1 systems a warp, the last size of the layout and the
    first past it; 37 systems leave a ragged warp.  The oracle's bound of the
    other least-squares tests."""
    _mgs_case(ht, L, 2, rows, cols, 37)


def _run(ht, s, L, m, predictor, **over):  # noqa: F811
    out = track_gpu(ht, s, L, m, h_min=1e-6, predictor=predictor, **over)
    return [np.asarray(v) for v in (out["x_end"], out["status"], out["t_end"], out["steps"])]


@pytest.mark.parametrize("L,n,deg,terms,few,many,predictor", [
    (1, 3, 2, 6, 3, 8, 0), (1, 6, 2, 8, 5, 64, 0), (1, 6, 2, 8, 5, 64, 2), (1, 8, 2, 10, 7, 256, 2), (1, 11, 2, 10, 9, 2048, 0),
    (1, 12, 2, 16, 33, 2000, 2), (1, 16, 2, 10, 17, 1500, 0), (1, 16, 2, 10, 17, 1500, 1), (1, 17, 2, 8, 5, 500, 0),
    (2, 3, 2, 6, 3, 8, 2), (2, 5, 2, 8, 5, 32, 0), (2, 9, 2, 10, 7, 512, 2), (2, 12, 2, 10, 33, 2600, 0),
    (2, 17, 2, 6, 3, 400, 0), (4, 4, 3, 8, 5, 81, 2), (4, 7, 2, 8, 6, 128, 1), (4, 10, 2, 8, 11, 1024, 2)])
def test_results_do_not_depend_on_the_number_of_paths(ht, L, n, deg, terms, few, many, predictor):  # noqa: F811
    """The first paths of a run by themselves (groups of one path, systems over
    all slots of a warp) and among many (larger groups, other layouts), and
    the last paths of the many one by one: the same bits."""
    s = synth.total_degree_system(900 + n, n, deg, terms)
    all_x, all_st, all_t, all_steps = _run(ht, s, L, many, predictor)
    x, st, t, steps = _run(ht, s, L, few, predictor)
    assert np.array_equal(x, all_x[..., :few]) and np.array_equal(st, all_st[:few])
    assert np.array_equal(t, all_t[:few]) and np.array_equal(steps, all_steps[:few])
    x, st, t, steps = _run(ht, s, L, 1, predictor, first=many - 1)
    assert np.array_equal(x[..., 0], all_x[..., -1]) and st[0] == all_st[-1] and t[0] == all_t[-1]
    assert steps[0] == all_steps[-1]
    assert np.mean(all_st == 1) > 0.5  # the comparison is of tracked paths
