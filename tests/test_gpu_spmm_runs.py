"""The tiled SpMM over slices of few tiles, which its blocks walk in runs of consecutive
tiles: the estimator's first pass with it against the plain SpMM."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _model(name, n, n_sys):
    if name == "xxz":
        return W.long_range_xxz(n, n_sys, 1.0, 0.7, 0.3, 0.8)
    if name == "chain":
        return W.xxz_chain(n, n_sys, 1.0, 0.5, 0.1)
    if name == "random":
        return W.random_model(n, n_sys, 5)
    if name == "tfim":
        return W.long_range_tfim(n, n_sys, 1.5, 0.9)
    # XX couplings of all pairs without YY: hops whose coefficient no row's parity changes
    # ("xx+x": with a transverse field on every other site)
    spec = W.long_range_xxz(n, n_sys, 1.2, 0.6, 0.2, 0.9)
    spec.jy[:] = 0.0
    if name == "xx+x":
        spec.gx[::2] = 0.45
    return spec


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


@pytest.mark.parametrize("model", ["xxz", "chain", "random", "tfim", "xx"])
@pytest.mark.parametrize("cols,dtype", [(8, "float32"), (4, "float64"), (4, "float32")])
def test_apply_keeps_infinities_to_coupled_rows(lib, model, cols, dtype):
    """H x with an infinity or a NaN in one row: it reaches the rows that H couples to that row
    (the non-zeros of H's column there) and no other, in the tiled kernel (32-byte rows) as in
    the plain one."""
    import torch
    n = 14
    spec = _model(model, n, 2)
    ctx = lib.Context(0)
    try:
        ham = lib.Hamiltonian(ctx, spec)
        for row in (0, 5, 777, 4099, 9999, 16383):
            x = torch.zeros(1 << n, cols, device="cuda", dtype=getattr(torch, dtype))
            y = torch.empty_like(x)
            x[row, 1] = 1.0
            ham.apply(x, y)
            torch.cuda.synchronize()
            coupled = y[:, 1] != 0
            coupled[row] = True  # (a vanishing diagonal element times the row itself)
            for bad in (float("inf"), float("nan")):
                x[row, 1] = bad
                ham.apply(x, y)
                torch.cuda.synchronize()
                assert torch.isfinite(y[:, 1][~coupled]).all()
                assert not torch.isfinite(y[:, 1][coupled & (torch.arange(1 << n, device="cuda") != row)]).any()
                assert torch.isfinite(y[:, [0, 2, 3]]).all()
    finally:
        ctx.close()


@pytest.mark.parametrize("n,n_sys,n_v,prec,tol", [
    (13, 0, 40, "fp32", 2e-5),
    (14, 2, 30, "fp32", 2e-5),
    (15, 1, 9, "fp32", 2e-5),
    (13, 1, 21, "fp64", 1e-12),
    (14, 2, 10, "fp64", 1e-12),
])
@pytest.mark.parametrize("model", ["xx", "xx+x"])
def test_uniform_hops_match_the_plain_spmm(lib, n, n_sys, n_v, prec, tol, model):
    """XX couplings of all pairs (c_odd = c_even) take the uniform instantiation with every kind
    of term: hops of register, row-group and high spins with one another, with and without
    fields. A_j and B_j of five steps against the plain SpMM, and rho against the oracle."""
    from oracle import lanczos
    spec = _model(model, n, n_sys)
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
        if n == 13:
            ref = lanczos.Estimator(spec).run(np.array([0.4]), n_v, 5, 31, "rademacher")
            np.testing.assert_allclose(out[1]["rho"], ref["rho"], atol=1e-4 if prec == "fp32" else 1e-10, rtol=0)
    finally:
        ctx.close()
