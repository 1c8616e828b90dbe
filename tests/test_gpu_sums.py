"""The float32 sums over the states behind T's coefficients: their rounding does not grow with
the rows one thread happens to take on a launch's grid."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

U = 2.0 ** -24  # float32's unit roundoff


def _rms_error(ham, n_v, key, j):
    """Relative rms distance of the float32 coefficients of step j from the float64 ones."""
    out = [ham.estimate([1.0], n_v, j + 1, 11, precision=p, dist="gauss", full=True)[key][:, j] for p in ("fp32", "fp64")]
    return np.sqrt(np.mean((out[0] - out[1]) ** 2) / np.mean(out[1] ** 2))


def test_qr_sums_of_many_vectors(lib):
    """2440 bath vectors are 610 slices: one block of the orthogonalisation per slice, 1024 rows
    a thread. A float32 sum over m rows of D rounds by about 0.15 u m / sqrt(D) of B_1: 0.42 u
    for m = 1024, 0.007 u for chains of 16; the vectors' own rounding (some 70 terms a row,
    independent over 2^17 rows) adds about 0.01 u."""
    ctx = lib.Context(0)
    try:
        ham = lib.Hamiltonian(ctx, W.long_range_xxz(17, 1, 1.0, 0.8, 0.3, 0.7))
        assert _rms_error(ham, 2440, "t_b", 0) < U / 8
    finally:
        ctx.close()


def test_projection_sums_of_runs_of_tiles(lib):
    """400 bath vectors of 2^16 states (d_s = 4) are 200 slices of 64 tiles, which the tiled SpMM
    walks in runs of several tiles. Against one vector alone, whose tiles are a block each, the
    rounding of A_1 is the same within the spread of an rms over that many coefficients."""
    ctx = lib.Context(0)
    try:
        ham = lib.Hamiltonian(ctx, W.long_range_xxz(16, 2, 1.0, 0.8, 0.3, 0.7))
        ctx.set_spmm_form(1)
        alone = []
        for l in range(40):
            out = [ham.estimate([1.0], 1, 1, 11, precision=p, dist="gauss", full=True, first_vector=l)["t_a"][:, 0]
                   for p in ("fp32", "fp64")]
            alone.append(np.mean((out[0] - out[1]) ** 2) / np.mean(out[1] ** 2))
        assert _rms_error(ham, 400, "t_a", 0) < 1.2 * np.sqrt(np.mean(alone))
    finally:
        ctx.close()
