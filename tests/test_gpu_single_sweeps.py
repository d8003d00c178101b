"""One sweep per call of the smallest lattices: byte planes for planes of at most one word, bit
streams from there, with the oracle's configurations, E and M call after call."""
import numpy as np
import pytest

import oracle
from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,L,R,n,kind", [
    (2, 2, 3, 1, "sweep_resident"), (2, 4, 200, 1, "sweep_resident"), (2, 8, 1, 1, "sweep_resident"),
    (2, 8, 5000, 1, "sweep_resident"), (2, 8, 10001, 1, "sweep_stream"), (2, 8, 1, 2, "sweep_stream"),
    (2, 10, 1, 1, "sweep_stream"), (3, 4, 3, 1, "sweep_stream"),
])
def test_single_sweeps(ctx, dim, L, R, n, kind):
    lat = gbmc.lattice_init(ctx, dim, L, n_replicas=R, seed=71)
    c = R - 1
    s = oracle.init_spins(dim, L, 71, 0, c, True)
    for call in range(3):
        E, M = device_i32(n * R), device_i32(n * R)
        gbmc.gbmc_profile(ctx, True)
        gbmc.metropolis_sweeps(ctx, lat, 0.4, n, *((E, M) if call else ()))
        prof = gbmc.gbmc_profile_read(ctx)
        gbmc.gbmc_profile(ctx, False)
        assert list(prof) == [kind], prof
        oracle.sweeps(dim, L, s, None, 0.4, 71, 0, c, n * call, n)
        np.testing.assert_array_equal(spins_out(ctx, lat)[c], s)
        if call:
            got = E.cpu().numpy().reshape(n, R)[-1, c], M.cpu().numpy().reshape(n, R)[-1, c]
            assert got == oracle.observables(dim, L, s, None)
    gbmc.lattice_free(lat)
