"""Populations with about one warp per scheduler, where two threads share a word of the
bit stream (each the sixteen sites of one half of it), against the byte-plane kernel: sizes whose
planes end in either half of their last word, with and without E and M after every sweep."""
import numpy as np
import pytest

from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu
FM, EA = gbmc.GBMC_ISING_FM, gbmc.GBMC_EA_PMJ


@pytest.mark.parametrize("dim,L,model,I,R,series", [
    (2, 24, FM, 1, 1513, False), (2, 30, FM, 1, 1100, False), (2, 10, FM, 1, 9000, False), (2, 64, FM, 1, 273, True),
    (2, 90, FM, 1, 160, True), (3, 6, EA, 3, 1345, False), (3, 10, EA, 2, 560, False), (3, 14, FM, 1, 300, False),
    (3, 16, EA, 1, 273, True),
])
def test_half_words_match_byte_kernel(ctx, dim, L, model, I, R, series):
    n, out = 4, []
    for kernel in (gbmc.GBMC_KERNEL_AUTO, gbmc.GBMC_KERNEL_BYTES):
        gbmc.gbmc_set_sweep_kernel(ctx, kernel)
        lat = gbmc.lattice_init(ctx, dim, L, model=model, n_instances=I, n_replicas=R, seed=70 + L, instance_base=1)
        E, M = (device_i32(n * I * R), device_i32(n * I * R)) if series else (None, None)
        gbmc.metropolis_sweeps(ctx, lat, 0.44 if dim == 2 else 0.5, n, E, M)
        out.append([spins_out(ctx, lat)] + ([E.cpu().numpy(), M.cpu().numpy()] if series else []))
        gbmc.lattice_free(lat)
    gbmc.gbmc_set_sweep_kernel(ctx, gbmc.GBMC_KERNEL_AUTO)
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
