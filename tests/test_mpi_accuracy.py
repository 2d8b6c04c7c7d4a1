"""Accuracy of the integer evaluation (csrc/ht_mpi_eval.cuh on the host) where
the terms of a sum differ in size: the accumulators' last limb, not the terms,
then limits the result."""
import ctypes

import numpy as np
import pytest

import synth
from parity import cerr
from test_mpi_host import _p, shim  # noqa: F401  (shim: the module's fixture)

# Units of 2^(-53 L) times the sum of an output's term moduli.  A term of the
# sum loses up to one unit of the frame's last place, 2^(E + 2 + head + 1) over
# the frame's width (29 (WA - 1) + 28 bits) with E the largest term's log2 and
# head the terms' bit count, so `terms` of them lose 2^(2 head + 3 - width):
# 2^-67, 2^-96 and 2^-212 for 246 terms in D (WA = 3), DD (4) and QD (8).  The
# conversion to L doubles cuts up to 2 units, a product of at most 5 factors
# and the derivative's exponent a few more; the two components' errors add as
# their root of squares.
UNITS = {1: 8.0, 2: 8.0 + 2.0 ** 10 * 1.5, 4: 8.0 + 1.5}


@pytest.mark.parametrize("L", [1, 2, 4])
@pytest.mark.parametrize("small", [1.0, 2.0 ** -20, 2.0 ** -45])
def test_sums_of_terms_of_different_sizes(oracle_lib, shim, L, small):  # noqa: F811
    """246 terms a polynomial, the first of modulus 1 and the others of modulus
    `small`, against the oracle with two (D) or L limbs."""
    shim.mpi_eval.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int] + [ctypes.c_void_p] * 3 + \
        [ctypes.c_int64] + [ctypes.c_void_p] * 3
    s = synth.config_system("pieri44_shape")
    first = np.concatenate([[0], np.cumsum(s.n_terms)[:-1]])
    scale = np.full((s.n_monomials, 1), small)
    scale[first] = 1.0
    s = synth.System(s.n_vars, s.n_polys, s.n_terms, s.exps, s.coef * scale)
    n = 3
    x = synth.unit_points(60 + L, s.n_vars, n, L)
    val = np.empty((s.n_polys, 2, L, n))
    jac = np.empty((s.n_polys, s.n_vars, 2, L, n))
    nt, ex = np.ascontiguousarray(s.n_terms, np.int32), np.ascontiguousarray(s.exps, np.int8)
    cf = s.coef_limbs(L)
    assert shim.mpi_eval(L, s.n_vars, s.n_polys, _p(nt), _p(ex), _p(cf), n, _p(x), _p(val), _p(jac)) == 0
    LO = max(L, 2)
    xo = np.zeros((s.n_vars, 2, LO, n))
    xo[:, :, :L] = x
    ref = oracle_lib.eval_(s, xo)
    mag = oracle_lib.eval_magnitude(s, x)
    for got, want, m in zip((val, jac), ref, mag):
        full = np.zeros_like(want)
        full[..., :L, :] = got
        units = cerr(full, want) / np.maximum(m, 1e-300) * 2.0 ** (53 * L)
        assert np.max(units) <= UNITS[L], (np.max(units), np.mean(units))
