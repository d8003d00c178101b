"""Large-lattice sweeps whose blocks hold their run of words in shared memory and read only
its ends from their neighbours: against the CPU oracle at the sizes on both sides of that rule
(runs hardly longer than their two ends, a run of the longest kind, runs that are whole
planes), with E and M after every sweep, and over many sweeps against the byte kernels."""
import numpy as np
import pytest

import oracle
from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu
INT8, BP = gbmc.GBMC_INT8, gbmc.GBMC_BITPACK


@pytest.mark.parametrize("L,R,layout,n", [(720, 1, INT8, 3), (760, 1, INT8, 3), (802, 1, INT8, 3), (896, 1, BP, 3),
                                          (1114, 1, INT8, 2), (1118, 1, INT8, 2), (520, 4, INT8, 3), (258, 14, INT8, 3),
                                          (64, 160, BP, 4), (64, 76, BP, 4)])
def test_held_runs_match_oracle(ctx, L, R, layout, n):
    seed = 300 + L
    lat = gbmc.lattice_init(ctx, 2, L, n_replicas=R, seed=seed, layout=layout)
    Es, Ms = device_i32(n * R), device_i32(n * R)
    gbmc.metropolis_sweeps(ctx, lat, 0.44, n, Es, Ms)
    got = spins_out(ctx, lat)
    Es, Ms = Es.cpu().numpy().reshape(n, R), Ms.cpu().numpy().reshape(n, R)
    for r in {0, R // 2, R - 1}:
        s = oracle.init_spins(2, L, seed, 0, r, True)
        for t in range(n):
            oracle.sweeps(2, L, s, None, 0.44, seed, 0, r, t, 1)
            assert (Es[t, r], Ms[t, r]) == oracle.observables(2, L, s, None), (r, t)
        np.testing.assert_array_equal(got[r], s)
    gbmc.lattice_free(lat)


@pytest.mark.parametrize("L,R", [(1000, 1), (760, 1), (520, 4)])
def test_held_runs_over_many_sweeps(ctx, L, R):
    out = []
    for kernel in (gbmc.GBMC_KERNEL_AUTO, gbmc.GBMC_KERNEL_BYTES):
        gbmc.gbmc_set_sweep_kernel(ctx, kernel)
        lat = gbmc.lattice_init(ctx, 2, L, n_replicas=R, seed=12)
        gbmc.metropolis_sweeps(ctx, lat, 0.44, 300)
        out.append(spins_out(ctx, lat))
        gbmc.lattice_free(lat)
    gbmc.gbmc_set_sweep_kernel(ctx, gbmc.GBMC_KERNEL_AUTO)
    np.testing.assert_array_equal(out[0], out[1])
