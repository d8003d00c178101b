"""Swendsen-Wang updates on every path (a block per copy on chip; tiles; the general kernels)
against the oracle's breadth-first labelling: labels, spins, E and M word for word, at sizes
where rows end inside a thread's four sites, at the largest lattices kept on chip and the next
ones, with one and many copies."""
import numpy as np
import pytest

import oracle
from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu
BC2, BC3 = 0.4406868, 0.2216544


@pytest.mark.parametrize("dim,L,R,n,beta,check", [
    # on chip
    (2, 4, 3, 8, BC2, (0, 2)), (2, 10, 2, 6, BC2, (0, 1)), (2, 14, 1, 6, 1.2, (0,)), (2, 30, 200, 4, BC2, (0, 199)),
    (2, 62, 2, 4, BC2, (1,)), (2, 126, 160, 2, BC2, (159,)), (2, 202, 152, 2, BC2, (3,)), (2, 50, 1, 3, 0.0, (0,)),
    (3, 4, 2, 6, BC3, (0, 1)), (3, 6, 3, 6, BC3, (2,)), (3, 10, 1, 6, 0.25, (0,)), (3, 18, 20, 3, BC3, (19,)),
    (3, 34, 200, 2, BC3, (7,)),
    # tiles
    (2, 64, 1200, 3, BC2, (0, 1199)), (2, 128, 1, 4, BC2, (0,)), (2, 160, 2, 3, 0.6, (1,)), (3, 32, 1, 3, BC3, (0,)),
    (3, 48, 1, 2, 0.3, (0,)), (2, 224, 1, 2, 0.0, (0,)),
    # tiles cut by the lattice's edge
    (2, 210, 1, 3, BC2, (0,)), (2, 250, 2, 2, 0.6, (1,)), (2, 164, 1, 3, BC2, (0,)), (2, 226, 1, 2, 1.2, (0,)),
    (2, 34, 9000, 2, BC2, (5, 8999)), (2, 36, 9000, 2, BC2, (8999,)), (2, 254, 1, 2, 0.0, (0,)),
    # neither
    (3, 34, 1, 2, BC3, (0,)), (3, 38, 1, 2, 0.3, (0,)), (2, 30, 30000, 2, BC2, (29999,)),
    (2, 2, 2, 4, BC2, (0, 1)),
])
def test_sw_sizes(ctx, dim, L, R, n, beta, check):
    seed = 7 + L
    lat = gbmc.lattice_init(ctx, dim, L, n_replicas=R, seed=seed, instance_base=1)
    N = L ** dim
    Es, Ms, labels = device_i32(n * R), device_i32(n * R), device_i32(R * N)
    Es.fill_(77)
    Ms.fill_(77)
    gbmc.swendsen_wang(ctx, lat, beta, n, Es, Ms, labels)
    got = spins_out(ctx, lat)
    Es, Ms = Es.cpu().numpy().reshape(n, R), Ms.cpu().numpy().reshape(n, R)
    labels = labels.cpu().numpy().reshape(R, N)
    for r in check:
        s = oracle.init_spins(dim, L, seed, 1, r, True)
        for u in range(n):
            lab = oracle.sw_update(dim, L, s, beta, seed, 1, r, u, want_labels=True)
            assert (Es[u, r], Ms[u, r]) == oracle.observables(dim, L, s), (r, u)
        np.testing.assert_array_equal(labels[r], lab)
        np.testing.assert_array_equal(got[r], s)
    gbmc.lattice_free(lat)
