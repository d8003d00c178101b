"""Bit-packed lattices that the row strips do not take: the launches per half-sweep read the bits as
they are and are the faster way for many sites and few sweeps, the strips beside tags for few sites,
many sweeps or E and M; the same configurations both ways."""
import numpy as np
import pytest

from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,R,n,series,kind", [
    (1088, 1, 2, False, "stream_strips"),
    (1984, 8, 4, False, "bitpack_halfsweep"),   # 31 million sites
    (1984, 8, 5, False, "stream_strips"),
    (4032, 4, 19, False, "bitpack_halfsweep"),  # 65 million
    (4032, 4, 20, False, "stream_strips"),
    (3008, 8, 20, False, "bitpack_halfsweep"),  # 72 million
    (3008, 8, 2, True, "stream_strips"),
])
def test_which_kernel_takes_them(ctx, L, R, n, series, kind):
    out = []
    for mode in (gbmc.GBMC_LAUNCH_AUTO, gbmc.GBMC_LAUNCH_GRID):
        gbmc.gbmc_set_sweep_launch(ctx, mode)
        try:
            lat = gbmc.lattice_init(ctx, 2, L, n_replicas=R, seed=51, layout=gbmc.GBMC_BITPACK)
            E, M = (device_i32(n * R), device_i32(n * R)) if series else (None, None)
            gbmc.gbmc_profile(ctx, True)
            gbmc.metropolis_sweeps(ctx, lat, 0.44, n, E, M)
            prof = gbmc.gbmc_profile_read(ctx)
            gbmc.gbmc_profile(ctx, False)
        finally:
            gbmc.gbmc_set_sweep_launch(ctx, gbmc.GBMC_LAUNCH_AUTO)
        want = kind if mode == gbmc.GBMC_LAUNCH_AUTO else "bitpack_halfsweep"
        assert want in prof and not {"stream_strips", "bitpack_halfsweep", "bitpack_strips"} & (set(prof) - {want}), prof
        out.append([spins_out(ctx, lat)] + ([E.cpu().numpy(), M.cpu().numpy()] if series else []))
        gbmc.lattice_free(lat)
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
