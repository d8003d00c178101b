"""Resampling of many small populations: beyond some hundred of them the grid-wide kernel takes a
lattice (a launch each), below it the clusters take all lattices in one launch; the same parents,
configurations and sums as one kernel per phase on both sides of the line."""
import numpy as np
import pytest

from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu
STEPS, R = 3, 39


def _run(ctx, fused, instances, law):
    gbmc.gbmc_set_resample_mode(ctx, fused)
    try:
        lats = [gbmc.lattice_init(ctx, 3, 4, model=gbmc.GBMC_EA_PMJ, n_instances=n, n_replicas=R, seed=7 + i)
                for i, n in enumerate(instances)]
        pa = gbmc.pa_create(ctx, lats, 1, STEPS, beta_f=0.6, resample=law, initial_replicas=12 if law else 0)
        gbmc.gbmc_profile(ctx, True)
        stats, _ = gbmc.pa_run(ctx, pa, capacity=STEPS + 1)
        prof = gbmc.gbmc_profile_read(ctx)
        gbmc.gbmc_profile(ctx, False)
        spins = [spins_out(ctx, l).reshape(n, R, -1) for l, n in zip(lats, instances)]
        gbmc.pa_free(pa)
        for l in lats:
            gbmc.lattice_free(l)
        return stats, spins, prof.get("pa_resample", (0, 0.0))[0]
    finally:
        gbmc.gbmc_set_resample_mode(ctx, True)


@pytest.mark.parametrize("law", [gbmc.GBMC_RESAMPLE_MULTINOMIAL, gbmc.GBMC_RESAMPLE_NEAREST,
                                 gbmc.GBMC_RESAMPLE_POISSON])
@pytest.mark.parametrize("instances,launches", [((100, 90), 1), ((101, 300), 2), ((600, 100), 2)])
def test_many_populations(ctx, law, instances, launches):
    a, sa, n = _run(ctx, True, instances, law)
    assert n == launches * STEPS
    b, sb, n = _run(ctx, False, instances, law)
    assert n == 0
    for f in ("sumE", "sumE2", "sumAbsM", "sumM2", "Emin", "Emax", "n_replicas"):
        np.testing.assert_array_equal(a[f], b[f], err_msg=f)
    np.testing.assert_allclose(a["lnZ"], b["lnZ"], rtol=1e-12, atol=1e-12)
    live = np.split(a["n_replicas"][STEPS], [instances[0]])
    for x, y, m in zip(sa, sb, live):
        for k, rows in enumerate(m):
            np.testing.assert_array_equal(x[k, :rows], y[k, :rows])
