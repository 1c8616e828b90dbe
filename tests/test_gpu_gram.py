"""The Gram form on a beta grid (float32, 32-byte rows): the betas run in groups inside one
launch, each group to the last step its betas need."""
import numpy as np
import pytest

import workloads as W
from oracle import lanczos

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_sys,n_v", [(10, 0, 3), (10, 1, 4), (11, 2, 2), (13, 2, 5), (12, 0, 9)])
@pytest.mark.parametrize("n_beta", [1, 2, 3, 5, 9, 17])
def test_gram_beta_groups(lib, n, n_sys, n_v, n_beta):
    """Each beta of a grid gives bit for bit what it gives alone (its psi and its sums do not
    depend on its group), in either order of the grid, with the basis stored or recomputed;
    and the values are the oracle's within the float32 contract."""
    spec = W.long_range_tfim(n, n_sys, 1.5, 0.8)
    betas = W.beta_grid(n_beta, 0.05, 6.0)
    ctx = lib.Context(0)
    try:
        ham = lib.Hamiltonian(ctx, spec)

        def run(b, **kw):
            return ham.estimate(b, n_v, 18, 77, precision="fp32", dist="gauss", full=True, **kw)
        ctx.set_device_dense(0)  # the same coefficients whatever the grid
        grid = run(betas)
        back = run(betas[::-1].copy())
        again = run(betas, passes="recompute")
        for i in range(n_beta):
            alone = run(betas[i:i + 1])
            np.testing.assert_array_equal(grid["gram_l"][i], alone["gram_l"][0])
            np.testing.assert_array_equal(grid["gram_l"][i], back["gram_l"][n_beta - 1 - i])
            np.testing.assert_array_equal(grid["gram_l"][i], again["gram_l"][i])
            g = grid["gram_l"][i]
            np.testing.assert_array_equal(g, np.swapaxes(g, 1, 2))
        ref = lanczos.Estimator(spec).run(betas, n_v, 18, 77, "gauss")
        np.testing.assert_allclose(grid["rho"], ref["rho"], atol=1e-4, rtol=0)
        np.testing.assert_allclose(grid["rho"], grid["rho_quad"], atol=1e-4, rtol=0)
    finally:
        ctx.close()


@pytest.mark.parametrize("n,n_sys,n_v,k", [(8, 1, 3, 1), (9, 0, 5, 7), (10, 2, 3, 40), (11, 1, 9, 33), (12, 2, 64, 12)])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_coefficients_on_the_device_are_the_hosts(lib, n, n_sys, n_v, k, prec):
    """With the basis stored, the Gram coefficients of a grid of 8 or more betas are formed
    on the device from the device small dense step; with the basis recomputed, on the host
    from the same step. The same products and sums in the same order: the same bits in the
    Gram and quadrature forms of every vector."""
    spec = W.random_model(n, n_sys, 17)
    ctx = lib.Context(0)
    try:
        ham = lib.Hamiltonian(ctx, spec)
        out = [ham.estimate(W.beta_grid(9, 0.02, 8.0), n_v, k, 4, precision=prec, dist="rademacher", full=True,
                            passes=p) for p in ("store", "recompute")]
        for key in ("quad_l", "gram_l", "rho", "lnZ", "rho_quad", "t_a", "t_b"):
            np.testing.assert_array_equal(out[0][key], out[1][key])
        slim = ham.estimate(W.beta_grid(9, 0.02, 8.0), n_v, k, 4, precision=prec, dist="rademacher")
        np.testing.assert_array_equal(slim["rho"], out[0]["rho"])
    finally:
        ctx.close()


@pytest.mark.parametrize("betas", [[14.0], [0.5, 11.0, 14.0, 18.0]])
@pytest.mark.parametrize("passes", ["store", "recompute"])
def test_gram_of_vectors_with_subnormal_weight(lib, betas, passes):
    """A diagonal H on basis vectors: psi_l is exp(-beta (E_l - E0) / 2) in one place, which runs
    through float32's subnormal numbers and out below them; the Gram of each vector is its
    square, within float32's spacing there (2^-149, half of it for each of two roundings) and
    the float32 rounding of the coefficient above."""
    spec = W.long_range_tfim(10, 0, 1.0, 0.0)
    ctx = lib.Context(0)
    try:
        ham = lib.Hamiltonian(ctx, spec)
        out = ham.estimate(betas, 1024, 1, 5, precision="fp32", dist="basis", full=True, passes=passes)
        e = out["t_a"][:, 0, 0, 0]
        subnormal = 0
        for bi, beta in enumerate(betas):
            psi = np.exp(-0.5 * beta * (e - e.min()))
            subnormal += int(np.sum((psi < 2.0 ** -126) & (psi > 2.0 ** -149)))
            np.testing.assert_array_less(np.abs(np.sqrt(out["gram_l"][bi, :, 0, 0]) - psi), 2.0 ** -149 + 4e-7 * psi)
        assert subnormal >= 10
    finally:
        ctx.close()


@pytest.mark.parametrize("n,n_sys,n_v,k,n_beta", [
    (12, 2, 3, 80, 9),    # groups of 2 betas (their coefficients pass 36 KB at 4)
    (12, 2, 3, 160, 3),   # groups of 1
    (12, 1, 3, 160, 5),   # d_s = 2, groups of 2
    (10, 0, 9, 6, 300),   # more betas than one launch takes
    (18, 0, 1, 6, 40),    # one slice: as many betas a launch as the partials have room for
])
def test_gram_groups_of_long_recurrences_and_grids(lib, n, n_sys, n_v, k, n_beta):
    """Each of a few betas of the grid gives bit for bit what it gives alone."""
    spec = W.xxz_chain(n, n_sys, 1.0, 0.5, 0.1)
    betas = W.beta_grid(n_beta, 0.05, 12.0)
    ctx = lib.Context(0)
    try:
        ham = lib.Hamiltonian(ctx, spec)
        ctx.set_device_dense(0)  # the same coefficients whatever the grid

        def run(b):
            return ham.estimate(b, n_v, k, 3, precision="fp32", dist="rademacher", full=True)
        grid = run(betas)
        for i in sorted({0, n_beta // 3, n_beta // 2, n_beta - 1}):
            np.testing.assert_array_equal(grid["gram_l"][i], run(betas[i:i + 1])["gram_l"][0])
        np.testing.assert_allclose(grid["rho"], grid["rho_quad"], atol=1e-4, rtol=0)
    finally:
        ctx.close()
