"""The waits of the sweeps of few small copies (updating warps for the bits that other warps draw
ahead) run out on purpose: a batch more than will come, a short cycle budget. The call
is reported, the next one is clean. The kernel that takes more copies than multiprocessors
has no such wait, so the same aid shows which of the two a call takes."""
import numpy as np
import pytest

import oracle
from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu
FM, EA = gbmc.GBMC_ISING_FM, gbmc.GBMC_EA_PMJ


def _phantom_status(ctx, lat, beta, n, E=None):
    gbmc.gbmc_test_barrier_wait(ctx, 1, 2_000_000)  # ~1 ms budget, one phantom batch
    try:
        gbmc.metropolis_sweeps(ctx, lat, beta, n, E)
        gbmc.gbmc_sync(ctx)
    except gbmc.GbmcError as e:
        return e.status
    finally:
        gbmc.gbmc_test_barrier_wait(ctx, 0, 2_000_000_000)
    return gbmc.GBMC_OK


# one updating warp and several, one batch of bits in all and many
@pytest.mark.parametrize("dim,L,model,R,n,series", [(2, 4, FM, 2, 2, False), (2, 16, FM, 1, 300, True),
                                                    (2, 90, FM, 2, 40, False), (3, 20, EA, 3, 10, True)])
def test_wait_runs_out_and_is_reported(ctx, dim, L, model, R, n, series):
    lat = gbmc.lattice_init(ctx, dim, L, model=model, n_replicas=R, seed=8)
    assert _phantom_status(ctx, lat, 0.44, n, device_i32(n * R) if series else None) == gbmc.GBMC_ERR_TIMEOUT
    gbmc.gbmc_sync(ctx)  # the flag was cleared when reported
    gbmc.lattice_free(lat)
    lat = gbmc.lattice_init(ctx, dim, L, model=model, n_replicas=R, seed=8)
    gbmc.metropolis_sweeps(ctx, lat, 0.44, 3)
    gbmc.gbmc_sync(ctx)
    s = oracle.init_spins(dim, L, 8, 0, R - 1, True)
    oracle.sweeps(dim, L, s, oracle.couplings(L, 8, 0) if model == EA else None, 0.44, 8, 0, R - 1, 0, 3)
    np.testing.assert_array_equal(spins_out(ctx, lat)[R - 1], s)
    gbmc.lattice_free(lat)


@pytest.mark.parametrize("dim,L,extra,n,status", [
    (2, 12, 0, 2, gbmc.GBMC_ERR_TIMEOUT), (2, 12, 1, 2, gbmc.GBMC_OK),   # a copy per multiprocessor, and one more
    (2, 12, 0, 1, gbmc.GBMC_OK),                                         # a single sweep
    (2, 90, 0, 2, gbmc.GBMC_ERR_TIMEOUT), (2, 92, 0, 2, gbmc.GBMC_OK),   # 127 and 133 words per plane
    (3, 20, 0, 2, gbmc.GBMC_ERR_TIMEOUT), (3, 22, 0, 2, gbmc.GBMC_OK),
])
def test_which_copies_have_their_bits_drawn_ahead(ctx, dim, L, extra, n, status):
    R = torch.cuda.get_device_properties(0).multi_processor_count + extra
    lat = gbmc.lattice_init(ctx, dim, L, n_replicas=R, seed=8)
    assert _phantom_status(ctx, lat, 0.3, n) == status
    gbmc.gbmc_sync(ctx)
    gbmc.lattice_free(lat)
