"""rdm_estimate_batch: uneven instances whose first passes share one persistent launch.

The estimator is a sum of independent recurrences (Sec. 3.1), so estimates of several
Hamiltonians can run side by side. Checks, through the C ABI:
  * every item of a mixed batch (different N, N_s, n_v, k, betas, precisions, vector
    distributions) matches the oracle (float64: 1e-10, float32: 1e-4 on rho*), and
    the same estimate run on its own through rdm_estimate (float64 items that take the
    untiled kernels: bit-identical; others within the precision contract);
  * an item's result is bit-identical alone (a batch of one) and in the mix;
  * the autotuner times its candidates once per size class and reuses the choice;
  * items the packed launch does not take (recomputed basis) run alongside.
"""
import numpy as np
import pytest

import workloads as W
from oracle import lanczos

pytestmark = pytest.mark.gpu


def _jobs(lib, ctx):
    specs = [
        (W.random_model(8, 2, 11), dict(n_v=3, k=12, seed=5, precision="fp64", dist="rademacher",
                                        betas=[0.5, 1.0])),
        (W.xxz_chain(10, 1, 1.0, 0.5), dict(n_v=16, k=40, seed=20220417, precision="fp64",
                                           dist="rademacher", betas=[0.5, 1.0, 2.0])),
        (W.long_range_tfim(11, 2, 1.5, 0.9), dict(n_v=5, k=25, seed=7, precision="fp32", dist="gauss",
                                                  betas=[1.0])),
        (W.random_model(9, 1, 3), dict(n_v=7, k=18, seed=9, precision="fp32", dist="rademacher",
                                       betas=[0.3, 3.0])),
        (W.long_range_xxz(12, 1, 1.0, 1.0, 0.1), dict(n_v=8, k=30, seed=13, precision="fp32",
                                                      dist="rademacher", betas=[0.7])),
        (W.random_model(7, 2, 4), dict(n_v=2, k=9, seed=17, precision="fp64", dist="gauss",
                                       betas=[1.5])),
    ]
    jobs = []
    for spec, kw in specs:
        jb = dict(kw)
        jb["ham"] = lib.Hamiltonian(ctx, spec)
        jb["spec"] = spec
        jobs.append(jb)
    return jobs


def test_batch_matches_oracle_and_single_estimates(lib):
    ctx = lib.Context(0)
    try:
        jobs = _jobs(lib, ctx)
        outs = ctx.estimate_batch(jobs)
        for jb, out in zip(jobs, outs):
            assert out["status"] == lib.OK
            tol = 1e-10 if jb["precision"] == "fp64" else 1e-4
            ref = lanczos.Estimator(jb["spec"]).run(jb["betas"], jb["n_v"], jb["k"], jb["seed"], jb["dist"])
            np.testing.assert_allclose(out["rho"], ref["rho"], atol=tol, rtol=0)
            single = jb["ham"].estimate(jb["betas"], jb["n_v"], jb["k"], jb["seed"], precision=jb["precision"],
                                        dist=jb["dist"])
            np.testing.assert_allclose(out["rho"], single["rho"], atol=tol, rtol=0)
            np.testing.assert_allclose(out["lnZ"], single["lnZ"], atol=1e3 * tol, rtol=0)
            if jb["precision"] == "fp64" and jb["spec"].n_sites < 10:  # both untiled: same arithmetic
                np.testing.assert_array_equal(out["rho"], single["rho"])
    finally:
        ctx.close()


def test_batch_item_alone_equals_in_mix(lib):
    ctx = lib.Context(0)
    try:
        jobs = _jobs(lib, ctx)
        mix = ctx.estimate_batch(jobs, full=True)
        for jb, m in zip(jobs, mix):
            alone = ctx.estimate_batch([jb], full=True)[0]
            for key in ("rho", "lnZ", "gram_l", "t_a", "t_b"):
                np.testing.assert_array_equal(alone[key], m[key])
        # order of the items in the batch does not matter either
        rev = ctx.estimate_batch(jobs[::-1])
        for a, b in zip(rev[::-1], mix):
            np.testing.assert_array_equal(a["rho"], b["rho"])
    finally:
        ctx.close()


def test_batch_autotuner_times_each_size_class_once(lib):
    ctx = lib.Context(0)
    try:
        jobs = _jobs(lib, ctx)
        assert ctx.packed_tuning() == (0, 0)
        ctx.estimate_batch(jobs)
        keys, runs = ctx.packed_tuning()
        assert keys >= 1 and runs >= keys
        ctx.estimate_batch(jobs)
        assert ctx.packed_tuning() == (keys, runs)
    finally:
        ctx.close()


def test_batch_with_items_outside_the_packed_launch(lib):
    ctx = lib.Context(0)
    try:
        jobs = _jobs(lib, ctx)[:3]
        jobs[1] = dict(jobs[1], passes="recompute")  # recomputed basis: runs as rdm_estimate does
        outs = ctx.estimate_batch(jobs)
        for jb, out in zip(jobs, outs):
            single = jb["ham"].estimate(jb["betas"], jb["n_v"], jb["k"], jb["seed"], precision=jb["precision"],
                                        dist=jb["dist"], passes=jb.get("passes", "auto"))
            tol = 1e-10 if jb["precision"] == "fp64" else 1e-4
            np.testing.assert_allclose(out["rho"], single["rho"], atol=tol, rtol=0)
    finally:
        ctx.close()


def test_batch_rejects_a_foreign_hamiltonian(lib):
    a, b = lib.Context(0), lib.Context(0)
    try:
        ham = lib.Hamiltonian(b, W.random_model(6, 1, 2))
        with pytest.raises(lib.RdmError) as e:
            a.estimate_batch([dict(ham=ham, betas=[1.0], n_v=2, k=4, seed=1)])
        assert e.value.status == lib.EINVAL
    finally:
        a.close()
        b.close()


def test_batch_device_dense_steps_in_one_launch(lib):
    """Items with 10-point beta grids take the device small dense step; a batch runs all
    their recurrences (both d_s groups) in one launch per d_s. Against each estimate on
    its own with the host path: float64 items within 1e-12 in rho*, float32 within the
    float32 contract."""
    ctx = lib.Context(0)
    try:
        jobs = _jobs(lib, ctx)
        for jb in jobs:
            jb["betas"] = list(W.beta_grid(10, 0.2, 6.0))
        ctx.profile(True)
        outs = ctx.estimate_batch(jobs)
        st = ctx.profile_stats()
        ctx.profile(False)
        assert st["dense_fT"]["launches"] == 2  # d_s = 2 and d_s = 4 groups
        ctx.set_device_dense(0)
        for jb, out in zip(jobs, outs):
            single = jb["ham"].estimate(jb["betas"], jb["n_v"], jb["k"], jb["seed"], precision=jb["precision"],
                                        dist=jb["dist"])
            tol = 1e-12 if jb["precision"] == "fp64" else 1e-4
            np.testing.assert_allclose(out["rho"], single["rho"], atol=tol, rtol=0)
    finally:
        ctx.close()


def test_batch_launch_forms_are_bit_identical(lib):
    """The packed first pass as the cooperative grid (grid barriers between phases) and
    as one block per slice (block barriers only): the same units with the same arithmetic,
    so every item's result is the same bit for bit; an unknown form is rejected."""
    ctx = lib.Context(0)
    try:
        jobs = _jobs(lib, ctx)
        outs = {}
        for form in (1, 2):
            ctx.set_packed_form(form)
            outs[form] = ctx.estimate_batch(jobs, full=True)
        for a, b in zip(outs[1], outs[2]):
            for key in ("rho", "lnZ", "gram_l", "t_a", "t_b"):
                np.testing.assert_array_equal(a[key], b[key])
        with pytest.raises(lib.RdmError) as e:
            ctx.set_packed_form(3)
        assert e.value.status == lib.EINVAL
    finally:
        ctx.close()


@pytest.mark.parametrize("n", [10, 11, 12, 13, 14])
@pytest.mark.parametrize("n_sys", [0, 1, 2])
def test_batch_first_passes_in_clusters(lib, n, n_sys):
    """float32 items of 2^10..2^14 states run their first pass in one thread-block cluster per
    slice (1 to 16 blocks): T's coefficients against the untiled units (form 1) over the
    first steps, within the float32 rounding of six steps; the whole estimate within the
    float32 contract; alone, in the mix and in another order bit for bit the same."""
    specs = [W.long_range_xxz(n, n_sys, 1.0, 0.8, 0.3, 0.7), W.random_model(n, n_sys, n),
             W.long_range_tfim(n, n_sys, 1.5, 0.9), W.xxz_chain(n, n_sys, 1.0, 0.5, 0.1)]
    ctx = lib.Context(0)
    try:
        jobs = [dict(ham=lib.Hamiltonian(ctx, s), betas=W.beta_grid(9, 0.1, 4.0), n_v=v, k=k, seed=40 + v,
                     precision="fp32", dist="gauss") for s, v, k in zip(specs, (1, 7, 16, 5), (18, 6, 25, 12))]
        mix = ctx.estimate_batch(jobs, full=True)
        rev = ctx.estimate_batch(jobs[::-1], full=True)[::-1]
        ctx.set_packed_form(1)
        plain = ctx.estimate_batch(jobs, full=True)
        ctx.set_packed_form(0)
        for jb, a, b, p in zip(jobs, mix, rev, plain):
            alone = ctx.estimate_batch([jb], full=True)[0]
            for key in ("rho", "lnZ", "gram_l", "t_a", "t_b"):
                np.testing.assert_array_equal(a[key], b[key])
                np.testing.assert_array_equal(a[key], alone[key])
            bound = jb["ham"].info()["norm_bound"]
            for key in ("t_a", "t_b"):
                np.testing.assert_allclose(a[key][:, :6], p[key][:, :6], atol=2e-5 * bound, rtol=0)
            np.testing.assert_allclose(a["rho"], p["rho"], atol=1e-4, rtol=0)
            np.testing.assert_allclose(a["rho"], a["rho_quad"], atol=1e-4, rtol=0)
    finally:
        ctx.close()


@pytest.mark.parametrize("n,n_sys,n_v", [(15, 2, 2), (15, 1, 4), (16, 2, 2)])
def test_many_small_items_are_no_slower_than_the_packed_launch(lib, n, n_sys, n_v):
    """Items of 32 tiles and up run their first passes by their own launches, side by side: 24
    of them of one slice each take no longer than in the packed launch (a quarter more is the
    margin for the clock), and each gives what it gives alone, bit for bit."""
    import time
    ctx = lib.Context(0)
    try:
        jobs = [dict(ham=lib.Hamiltonian(ctx, W.xxz_chain(n, n_sys, 1.0, 0.3 + 0.02 * i, 0.1)), betas=[1.0], n_v=n_v,
                     k=20, seed=i, precision="fp32") for i in range(24)]
        ms = []
        for form in (0, 1, 2):
            ctx.set_packed_form(form)
            best = 1e9
            for _ in range(6):
                t0 = time.perf_counter()
                out = ctx.estimate_batch(jobs, full=True)
                best = min(best, time.perf_counter() - t0)
            ms.append(1e3 * best)
            if form == 0:
                mix = out
        assert ms[0] < 1.25 * min(ms[1:]), ms
        ctx.set_packed_form(0)
        for jb, a in list(zip(jobs, mix))[::6]:
            alone = ctx.estimate_batch([jb], full=True)[0]
            for key in ("rho", "lnZ", "gram_l", "t_a", "t_b"):
                np.testing.assert_array_equal(a[key], alone[key])
    finally:
        ctx.close()


def test_plain_spmm_form_holds_in_batches(lib):
    """rdm_set_spmm_form(2) asks for the plain SpMM: a batch's small float32 items then run the
    packed launch's plain units (bit for bit those of rdm_set_packed_form(1)), not the tiled
    arithmetic of the clusters."""
    ctx = lib.Context(0)
    try:
        jobs = [dict(ham=lib.Hamiltonian(ctx, W.random_model(n, 1, n)), betas=[0.5], n_v=3, k=6, seed=9,
                     precision="fp32") for n in (10, 12, 13)]
        ctx.set_packed_form(1)
        units = ctx.estimate_batch(jobs, full=True)
        ctx.set_packed_form(0)
        ctx.set_spmm_form(2)
        plain = ctx.estimate_batch(jobs, full=True)
        for a, b in zip(units, plain):
            for key in ("rho", "t_a", "t_b"):
                np.testing.assert_array_equal(a[key], b[key])
    finally:
        ctx.close()


def test_batch_of_every_launch(lib):
    """One item for each launch a batch can have (clusters by d_s and size, packed launches by
    precision and d_s), with many steps each: the launches' descriptors lie one behind the
    other, and every item gives what it gives alone, bit for bit."""
    ctx = lib.Context(0)
    try:
        jobs = [dict(ham=lib.Hamiltonian(ctx, W.long_range_tfim(n, s, 1.5, 0.9)), betas=[0.7], n_v=2, k=60 + 5 * s + n,
                     seed=n, precision=p) for s in (0, 1, 2)
                for n, p in ((10, "fp32"), (11, "fp32"), (12, "fp32"), (13, "fp32"), (14, "fp32"), (8, "fp32"), (9, "fp64"))]
        mix = ctx.estimate_batch(jobs, full=True)
        for jb, a in zip(jobs, mix):
            alone = ctx.estimate_batch([jb], full=True)[0]
            for key in ("rho", "lnZ", "gram_l", "t_a", "t_b"):
                np.testing.assert_array_equal(a[key], alone[key])
    finally:
        ctx.close()


def test_cluster_launches_run_side_by_side(lib):
    """Four items of one slice each, of four sizes: four cluster launches, which take a fraction
    of the GPU each and run at the same time. Timed launches (the profile) run one after
    another; untimed, the batch takes that less the sum of their times, and the longest of
    them more (with half of that as the margin)."""
    import time
    ctx = lib.Context(0)
    try:
        jobs = [dict(ham=lib.Hamiltonian(ctx, W.long_range_xxz(n, 0, 1.0, 0.8)), betas=[0.5], n_v=1, k=400, seed=3,
                     precision="fp32") for n in (10, 11, 12, 13)]

        def clock(batch):
            best = 1e9
            for _ in range(8):
                t0 = time.perf_counter()
                ctx.estimate_batch(batch)
                best = min(best, time.perf_counter() - t0)
            return 1e3 * best

        def first_pass(batch):
            ctx.profile(True)
            ctx.estimate_batch(batch)
            ms = ctx.profile_stats()["packed_pass1"]["ms"]
            ctx.profile(False)
            return ms

        clock(jobs)
        each = [first_pass([jb]) for jb in jobs]
        ctx.profile(True)
        serial = clock(jobs)
        ctx.profile(False)
        assert clock(jobs) < serial - sum(each) + 1.5 * max(each), (serial, each)
    finally:
        ctx.close()


@pytest.mark.parametrize("n,n_sys", [(13, 0), (14, 1), (14, 2)])
@pytest.mark.parametrize("field", [0.0, 0.45])
def test_uniform_hops_in_clusters(lib, n, n_sys, field):
    """XX couplings of all pairs (no parity-dependent coefficient) through the cluster pass,
    against the packed launch's plain units, within the float32 rounding of six steps."""
    spec = W.long_range_xxz(n, n_sys, 1.2, 0.6, 0.2, 0.9)
    spec.jy[:] = 0.0
    spec.gx[::2] = field
    ctx = lib.Context(0)
    try:
        job = dict(ham=lib.Hamiltonian(ctx, spec), betas=[0.4], n_v=5, k=6, seed=2, precision="fp32")
        a = ctx.estimate_batch([job], full=True)[0]
        ctx.set_packed_form(1)
        b = ctx.estimate_batch([job], full=True)[0]
        for key in ("t_a", "t_b"):
            np.testing.assert_allclose(a[key], b[key], atol=2e-5 * job["ham"].info()["norm_bound"], rtol=0)
    finally:
        ctx.close()
