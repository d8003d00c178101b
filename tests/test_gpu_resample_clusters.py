"""Resampling of a population in one cluster of blocks against one kernel per phase (the
general path): the same parents and populations, so the same configurations and integer
sums word for word; ln Z sums the same terms in another tree (a few hundred positive
terms, 1e-13 relative per step)."""
import numpy as np
import pytest

import oracle

from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu

LAWS = {"multinomial": gbmc.GBMC_RESAMPLE_MULTINOMIAL, "nearest": gbmc.GBMC_RESAMPLE_NEAREST,
        "poisson": gbmc.GBMC_RESAMPLE_POISSON}
STEPS = 4


def _run(ctx, fused, sizes, law, instances, start, L):
    gbmc.gbmc_set_resample_mode(ctx, fused)
    try:
        lats = [gbmc.lattice_init(ctx, 2, L, n_instances=instances, n_replicas=R, seed=7 + i)
                for i, R in enumerate(sizes)]
        pa = gbmc.pa_create(ctx, lats, 1, STEPS, beta_f=0.5, resample=LAWS[law], initial_replicas=start)
        stats, n = gbmc.pa_run(ctx, pa, capacity=STEPS + 1)
        assert n == STEPS
        out = dict(stats=stats, spins=[spins_out(ctx, l) for l in lats], parents=[])
        for i, R in enumerate(sizes):
            par = np.zeros(instances * R, dtype=np.uint32)
            gbmc.pa_parents_out(ctx, pa, i, par)
            out["parents"].append(par.reshape(instances, R))
        gbmc.pa_free(pa)
        for l in lats:
            gbmc.lattice_free(l)
        return out
    finally:
        gbmc.gbmc_set_resample_mode(ctx, True)


def _compare(ctx, sizes, law, instances=1, start=0):
    L = 8 if len(sizes) == 1 else 32  # (a run's 8 x 8 lattices need populations alike)
    a, b = (_run(ctx, fused, sizes, law, instances, start, L) for fused in (True, False))
    for f in ("sumE", "sumE2", "sumAbsM", "sumM2", "Emin", "Emax", "n_replicas", "step"):
        np.testing.assert_array_equal(a["stats"][f], b["stats"][f], err_msg=f)
    for f in ("lnQ", "lnZ"):
        np.testing.assert_allclose(a["stats"][f], b["stats"][f], rtol=1e-12, atol=1e-12, err_msg=f)
    live = a["stats"]["n_replicas"][STEPS]
    pop = 0
    for i, R in enumerate(sizes):
        for k in range(instances):
            n = int(live[pop])
            np.testing.assert_array_equal(a["parents"][i][k, :n], b["parents"][i][k, :n])
            np.testing.assert_array_equal(a["spins"][i][k * R:k * R + n], b["spins"][i][k * R:k * R + n])
            pop += 1


# slices of 7 or 15 workers, their edges, runs of several replicas per thread, and both
# sides of the rule's line
@pytest.mark.parametrize("R", [1, 2, 6, 7, 8, 63, 513, 2048, 2049, 7 * 512 + 1, 15 * 512 - 1, 15 * 512 + 16, 24576, 24577])
def test_multinomial(ctx, R):
    _compare(ctx, [R], "multinomial")


@pytest.mark.parametrize("law,R,start", [("nearest", 40, 10), ("nearest", 2049, 1500), ("nearest", 65536, 60000),
                                         ("nearest", 65537, 60000), ("poisson", 60, 10), ("poisson", 700, 500),
                                         ("poisson", 8192, 7000), ("poisson", 8193, 7000)])
def test_variable_populations(ctx, law, R, start):
    _compare(ctx, [R], law, start=start)


@pytest.mark.parametrize("sizes,instances", [([300], 5), ([4000], 4), ([4000], 6), ([100], 40), ([24576], 9),
                                             ([1000, 30, 5000], 1), ([24576, 24577, 9], 2)])
def test_several_populations_in_one_launch(ctx, sizes, instances):
    _compare(ctx, sizes, "multinomial", instances=instances)


# one step so large that a replica or two take the whole population: Poisson means of hundreds
# (past the tabulated inverses) and, above 500, in pieces
@pytest.mark.parametrize("R0,cap", [(450, 900), (900, 1500), (2100, 2800)])
def test_poisson_with_large_means(ctx, R0, cap):
    L, S, theta, seed = 32, 1, 1, 31
    lat = gbmc.lattice_init(ctx, 2, L, n_replicas=cap, seed=seed)
    pa = gbmc.pa_create(ctx, [lat], theta, S, beta_f=1.0, resample=LAWS["poisson"], initial_replicas=R0)
    stats, n = gbmc.pa_run(ctx, pa, capacity=S + 1)
    ref = oracle.pa_run_nearest(2, L, seed, 0, R0, cap, oracle.linear_betas(1.0, S), theta, poisson=True)
    assert n == S and ref["ok"]
    live = int(ref["nrep"][-1])
    par = np.empty(cap, dtype=np.uint32)
    gbmc.pa_parents_out(ctx, pa, 0, par)
    np.testing.assert_array_equal(stats["n_replicas"][:, 0], ref["nrep"])
    np.testing.assert_array_equal(par[:live], ref["parents"])
    assert np.bincount(par[:live]).max() > 0.3 * R0  # such a mean did occur
    gbmc.pa_free(pa)
    gbmc.lattice_free(lat)
