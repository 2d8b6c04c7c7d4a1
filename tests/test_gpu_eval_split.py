"""Evaluation of few points: polynomials split over several warps give the
bits of the unsplit kernels."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ht():
    from paper_1505_00383_gb300 import _build, ht as binding
    _build.build()
    assert torch.cuda.is_available()
    return binding


def _eval(ht, system, L, x, variant, threads):
    hs = ht.system_from(system, L)
    ht.ht_set_eval_config(hs, variant, threads)
    n = x.shape[-1]
    xd = torch.from_numpy(x).cuda()
    val = torch.full((system.n_polys, 2, L, n), float("nan"), dtype=torch.float64, device="cuda")
    jac = torch.full((system.n_polys, system.n_vars, 2, L, n), float("nan"), dtype=torch.float64, device="cuda")
    ht.ht_eval_diff(hs, n, xd, val, jac)
    torch.cuda.synchronize()
    return val.cpu().numpy(), jac.cpu().numpy()


@pytest.mark.parametrize("L", [1, 2, 4])
@pytest.mark.parametrize("name,n", [("cyclic10_shape", 1), ("cyclic10_shape", 33), ("nash8_shape", 31),
                                    ("pieri44_shape", 999), ("pieri44_shape", 3001), ("evaldiff_n32", 70),
                                    ("extreme", 40)])
def test_integer_split_matches_the_unit_kernel(ht, name, n, L):
    """Splits of 1 to 16 warps a polynomial (one point to several waves of CTAs,
    ragged last blocks, polynomials of 2 to 246 monomials, 64-variable monomials and x^127) against the per-unit
    kernel, which never splits: exact sums, so the same bits."""
    s = synth.extreme_system(3, 64, 5) if name == "extreme" else synth.config_system(name)
    x = synth.unit_points(41, s.n_vars, n, L)
    x[:, :, :, n // 2] *= 1e-30  # terms of very different sizes in one block
    x[s.n_vars // 2, :, :, 0] = 0.0
    for got, ref in zip(_eval(ht, s, L, x, 2, 256), _eval(ht, s, L, x, 2, 128)):
        assert np.array_equal(got, ref)


@pytest.mark.parametrize("name,n", [("cyclic10_shape", 1), ("cyclic10_shape", 33), ("nash8_shape", 31),
                                    ("pieri44_shape", 999), ("pieri44_shape", 3001), ("evaldiff_n32", 70),
                                    ("plain_n6_d", 5), ("extreme", 40)])
def test_double_split_matches_the_unrolled_bodies(ht, name, n):
    """The default kernel at few points (monomials over the warps of a CTA, the
    terms of 246 monomials in chunks) against variant 0, which never splits:
    the same operations in the same order, so the same bits."""
    s = synth.extreme_system(3, 64, 5) if name == "extreme" else synth.config_system(name)
    x = synth.unit_points(43, s.n_vars, n, 1)
    x[s.n_vars // 2, :, :, 0] = 0.0
    ref = _eval(ht, s, 1, x, 0, 0)
    for variant in (-1, 1):
        for got, want in zip(_eval(ht, s, 1, x, variant, 0), ref):
            assert np.array_equal(got, want)
