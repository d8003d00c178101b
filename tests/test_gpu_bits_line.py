"""The line between the bit-sliced kernel and the bit stream lies lower for a single sweep, whose way
in and out of the bits counts most: the kernel that takes each side, and the oracle's copies."""
import numpy as np
import pytest

import oracle
from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,L,R,n,kind", [
    (2, 64, 300, 1, "sweep_stream"), (2, 64, 600, 1, "sweep_bits"), (2, 64, 600, 3, "sweep_stream"),
    (2, 128, 900, 1, "sweep_stream"), (2, 128, 1300, 1, "sweep_bits"), (2, 128, 2400, 2, "sweep_stream"),
    (2, 256, 1800, 1, "sweep_stream"), (2, 256, 1900, 1, "sweep_bits"), (2, 256, 2600, 2, "sweep_bits"),
    (2, 256, 2600, 3, "sweep_stream"), (3, 16, 400, 1, "sweep_stream"), (3, 16, 600, 1, "sweep_bits"),
])
def test_which_side(ctx, dim, L, R, n, kind):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the line is for 152 multiprocessors")
    lat = gbmc.lattice_init(ctx, dim, L, n_replicas=R, seed=81)
    gbmc.gbmc_profile(ctx, True)
    gbmc.metropolis_sweeps(ctx, lat, 0.4, n)
    prof = gbmc.gbmc_profile_read(ctx)
    gbmc.gbmc_profile(ctx, False)
    assert list(prof) == [kind], prof
    got = spins_out(ctx, lat)
    for c in (0, R - 1):
        s = oracle.init_spins(dim, L, 81, 0, c, True)
        oracle.sweeps(dim, L, s, None, 0.4, 81, 0, c, 0, n)
        np.testing.assert_array_equal(got[c], s)
    gbmc.lattice_free(lat)
