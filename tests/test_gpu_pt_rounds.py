"""Rounds of parallel tempering in one launch against one sweep and one exchange launch per
round (BITS mode, the general path): configurations, maps, accepted swaps and energies word for
word, over the ways an instance is divided (a warp's share of copies, whole blocks, clusters
whose last blocks hold nothing) and several calls in a row."""
import numpy as np
import pytest

from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu
FM, EA = gbmc.GBMC_ISING_FM, gbmc.GBMC_EA_PMJ


def _run(ctx, kernel, dim, L, model, I, T, theta, calls):
    lat = gbmc.lattice_init(ctx, dim, L, model=model, n_instances=I, n_replicas=T, seed=5, instance_base=1)
    pt = gbmc.pt_create(ctx, lat, np.linspace(0.2, 1.2 if model == EA else 0.6, T), theta)
    gbmc.gbmc_set_sweep_kernel(ctx, kernel)
    gbmc.gbmc_profile(ctx, True)
    try:
        for n in calls:
            gbmc.pt_step(ctx, pt, n)
        names = set(gbmc.gbmc_profile_read(ctx))
    finally:
        gbmc.gbmc_profile(ctx, False)
        gbmc.gbmc_set_sweep_kernel(ctx, gbmc.GBMC_KERNEL_AUTO)
    rep, E = np.empty(I * T, dtype=np.uint32), np.empty(I * T, dtype=np.int32)
    acc = np.empty(I * max(T - 1, 1), dtype=np.uint32)
    gbmc.pt_state_out(ctx, pt, rep, acc if T > 1 else None, E)
    gbmc.pt_free(pt)
    out = spins_out(ctx, lat), rep, acc if T > 1 else None, E
    gbmc.lattice_free(lat)
    return out, names


@pytest.mark.parametrize("dim,L,model,I,T,theta,calls", [
    (3, 8, EA, 40, 32, 2, (3, 1, 2)),    # four copies per warp
    (3, 4, EA, 3, 40, 1, (1, 4)),        # one word per plane
    (3, 4, FM, 1, 2, 3, (5,)),           # one pair
    (3, 6, EA, 160, 9, 1, (4,)),         # partly filled last warps
    (3, 10, FM, 2, 13, 2, (3, 2)),       # blocks of a cluster with fewer copies than the others
    (3, 12, EA, 100, 36, 1, (3,)),       # whole-block teams, more blocks than places
    (3, 16, EA, 3, 11, 1, (3,)),
    (2, 6, FM, 4, 5, 2, (7,)),
    (2, 24, FM, 30, 17, 1, (4,)),
    (2, 64, FM, 2, 8, 2, (3,)),
    (3, 8, FM, 2, 700, 1, (2,)),         # more temperatures than threads
])
def test_rounds_match_single_launches(ctx, dim, L, model, I, T, theta, calls):
    a, names = _run(ctx, gbmc.GBMC_KERNEL_AUTO, dim, L, model, I, T, theta, calls)
    b, plain = _run(ctx, gbmc.GBMC_KERNEL_BITS, dim, L, model, I, T, theta, calls)
    assert "pt_rounds" in names and "pt_rounds" not in plain
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)
