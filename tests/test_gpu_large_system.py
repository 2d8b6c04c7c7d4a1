"""A system whose sweep steps outnumber 32-bit offsets (host lists only: it is
evaluated at a handful of points)."""
import numpy as np
import pytest

from test_gpu_track import ht  # noqa: F401  (the module's fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_system_past_the_step_offsets_evaluates_on_the_fp64_bodies(ht):  # noqa: F811
    """2,040 polynomials of 128 monomials in 64 variables of exponent 127: 2.16
    billion steps.  Creation builds no step list, and the integer variant falls
    back to the FP64 bodies' bits."""
    np_, terms, nv, n = 2040, 128, 64, 2
    rng = np.random.default_rng(8)
    M = np_ * terms
    th = rng.uniform(0, 2 * np.pi, M)
    coef = np.ascontiguousarray(np.stack([np.cos(th), np.sin(th)], axis=1))[:, :, None]
    hs = ht.ht_create_system(nv, np_, np.full(np_, terms, np.int32), np.full((M, nv), 127, np.int8), coef, 1)
    ph = torch.rand((nv, n), dtype=torch.float64, device="cuda") * 6.28
    x = torch.stack([torch.cos(ph), torch.sin(ph)], dim=1)[:, :, None].contiguous()
    out = []
    for variant, threads in ((0, 0), (2, 256), (2, 128)):
        ht.ht_set_eval_config(hs, variant, threads)
        val = torch.full((np_, 2, 1, n), float("nan"), dtype=torch.float64, device="cuda")
        jac = torch.full((np_, nv, 2, 1, n), float("nan"), dtype=torch.float64, device="cuda")
        ht.ht_eval_diff(hs, n, x, val, jac)
        torch.cuda.synchronize()
        out.append((val.cpu().numpy(), jac.cpu().numpy()))
    assert np.all(np.isfinite(out[0][0])) and np.all(np.isfinite(out[0][1]))
    for o in out[1:]:
        assert np.array_equal(o[0], out[0][0]) and np.array_equal(o[1], out[0][1])
    # sum of 128 terms of modulus one
    assert np.max(np.hypot(out[0][0][:, 0], out[0][0][:, 1])) <= 128.5
