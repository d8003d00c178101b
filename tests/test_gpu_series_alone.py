"""E alone, M alone and both together give the same series in every kernel that a sweep call can
take: byte planes, bit-sliced, bit streams, bits drawn ahead, strips, halo tiles, launches per
half-sweep, the bit-packed layout, double checkerboard, cluster updates."""
import numpy as np
import pytest

from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu
FM, EA, INT8, BP = gbmc.GBMC_ISING_FM, gbmc.GBMC_EA_PMJ, gbmc.GBMC_INT8, gbmc.GBMC_BITPACK
AUTO, BYTES, BITS = gbmc.GBMC_KERNEL_AUTO, gbmc.GBMC_KERNEL_BYTES, gbmc.GBMC_KERNEL_BITS
N = 3


@pytest.mark.parametrize("dim,L,model,layout,R,kernel,launch,how", [
    (2, 8, FM, INT8, 3, BYTES, 0, "sweeps"), (2, 10, FM, INT8, 3, BYTES, 0, "sweeps"), (3, 8, EA, INT8, 2, BYTES, 2, "sweeps"),
    (2, 8, FM, INT8, 500, AUTO, 0, "sweeps"), (2, 64, FM, INT8, 5, BITS, 0, "sweeps"), (3, 8, EA, INT8, 5, BITS, 0, "sweeps"),
    (2, 16, FM, INT8, 9, BITS, 0, "sweeps"), (2, 24, FM, INT8, 2, AUTO, 0, "sweeps"), (2, 24, FM, INT8, 3000, AUTO, 0, "sweeps"),
    (2, 520, FM, INT8, 1, AUTO, 0, "sweeps"), (2, 512, FM, INT8, 1, AUTO, 1, "sweeps"), (2, 520, FM, INT8, 1, AUTO, 1, "sweeps"),
    (3, 66, EA, INT8, 1, AUTO, 1, "sweeps"), (2, 128, FM, BP, 2, AUTO, 0, "sweeps"), (2, 128, FM, BP, 2, AUTO, 1, "sweeps"),
    (2, 128, FM, INT8, 2, AUTO, 0, "dcb"), (2, 64, FM, INT8, 2, BYTES, 0, "dcb"), (2, 16, FM, INT8, 2, AUTO, 0, "sw"),
    (2, 258, FM, INT8, 1, AUTO, 0, "sw"),
])
def test_one_series_alone(ctx, dim, L, model, layout, R, kernel, launch, how):
    out = []
    gbmc.gbmc_set_sweep_kernel(ctx, kernel)
    gbmc.gbmc_set_sweep_launch(ctx, launch)
    try:
        for want in ("EM", "E", "M"):
            lat = gbmc.lattice_init(ctx, dim, L, model=model, n_replicas=R, seed=61, layout=layout)
            E, M = (device_i32(N * R) + 7 if k in want else None for k in "EM")
            if how == "sw":
                gbmc.swendsen_wang(ctx, lat, 0.4, N, E, M)
            elif how == "dcb":
                gbmc.metropolis_sweeps_dcb(ctx, lat, 0.4, N, 1, 32, E, M)
            else:
                gbmc.metropolis_sweeps(ctx, lat, 0.4, N, E, M)
            gbmc.gbmc_sync(ctx)
            out.append((spins_out(ctx, lat), *(None if x is None else x.cpu().numpy() for x in (E, M))))
            gbmc.lattice_free(lat)
    finally:
        gbmc.gbmc_set_sweep_kernel(ctx, AUTO)
        gbmc.gbmc_set_sweep_launch(ctx, 0)
    for alone in out[1:]:
        for a, b in zip(out[0], alone):
            if b is not None:
                np.testing.assert_array_equal(a, b)
