"""The tiled SpMM over slices of few tiles, which its blocks walk in runs of consecutive
tiles: the estimator's first pass with it against the plain SpMM."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_sys,n_v,prec,tol", [
    (10, 2, 640, "fp32", 2e-5),   # one tile per slice
    (11, 2, 333, "fp64", 1e-12),  # two, a padded last slice in float32 only
    (11, 1, 801, "fp32", 2e-5),
    (13, 2, 301, "fp32", 2e-5),   # eight: a run is a slice
    (14, 1, 97, "fp64", 1e-12),
    (14, 0, 500, "fp32", 2e-5),
])
@pytest.mark.parametrize("model", ["xxz", "random", "tfim"])
def test_runs_of_tiles_match_the_plain_spmm(lib, n, n_sys, n_v, prec, tol, model):
    """A_j and B_j of five Lanczos steps, relative to the norm bound of H: the tolerance is
    the vectors' rounding (u per product of about 100 terms, five steps)."""
    spec = {"xxz": lambda: W.long_range_xxz(n, n_sys, 1.0, 0.7, 0.3, 0.8),
            "random": lambda: W.random_model(n, n_sys, 5),
            "tfim": lambda: W.long_range_tfim(n, n_sys, 1.5, 0.9)}[model]()
    ctx = lib.Context(0)
    try:
        ham = lib.Hamiltonian(ctx, spec)
        out = {}
        for form in (1, 2):
            ctx.set_spmm_form(form)
            out[form] = ham.estimate([0.4], n_v, 5, 31, precision=prec, dist="rademacher", full=True)
        bound = ham.info()["norm_bound"]
        for key in ("t_a", "t_b"):
            np.testing.assert_allclose(out[1][key], out[2][key], atol=tol * bound, rtol=0)
        np.testing.assert_allclose(out[1]["rho"], out[2]["rho"], atol=tol, rtol=0)
    finally:
        ctx.close()
