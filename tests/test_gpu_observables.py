"""E and M of whole configurations (one kernel over words or 16-site chunks, one or
several blocks per copy) and the int8 <-> bit-packed conversion, against numpy."""
import numpy as np
import pytest

import oracle
from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu

FM, EA, BP = gbmc.GBMC_ISING_FM, gbmc.GBMC_EA_PMJ, gbmc.GBMC_BITPACK


def _numpy_observables(dim, L, s, J):
    """E (forward bonds) and M of copies s [C][N]; J [C][N][dim] or None."""
    s = s.reshape(-1, *([L] * dim)).astype(np.int64)
    E = np.zeros(len(s), dtype=np.int64)
    for mu in range(dim):
        bond = s * np.roll(s, -1, axis=dim - mu)
        if J is not None:
            bond = bond * J[..., mu].reshape(s.shape)
        E -= bond.reshape(len(s), -1).sum(1)
    return E, s.reshape(len(s), -1).sum(1)


@pytest.mark.parametrize("dim,L,model,I,R", [
    (2, 2, FM, 1, 3), (2, 4, FM, 2, 5), (2, 6, FM, 1, 70), (2, 10, FM, 3, 33), (2, 16, FM, 2, 19), (2, 18, FM, 1, 9),
    (2, 48, FM, 1, 5), (2, 100, FM, 1, 3), (2, 258, FM, 1, 1), (2, 1000, FM, 1, 2), (2, 1024, FM, 1, 1),
    (2, 8, FM, 1, 70000),   # more copies than one launch takes blocks
    (3, 2, EA, 2, 3), (3, 4, EA, 3, 5), (3, 6, EA, 2, 9), (3, 10, FM, 1, 3), (3, 16, EA, 2, 2), (3, 18, EA, 1, 2),
    (3, 48, EA, 2, 1), (3, 50, EA, 1, 1), (3, 64, FM, 1, 1),
])
def test_observables_match_numpy(ctx, dim, L, model, I, R):
    lat = gbmc.lattice_init(ctx, dim, L, model=model, n_instances=I, n_replicas=R, seed=5 + L)
    E, M = device_i32(I * R) + 7, device_i32(I * R) - 3  # overwritten, not added to
    gbmc.observables(ctx, lat, E, M)
    s = spins_out(ctx, lat)
    J = None
    if model == EA:
        J = gbmc.lattice_couplings_out(ctx, lat, np.empty((I, L ** dim, 3), dtype=np.int8)).astype(np.int64)
        J = np.repeat(J, R, axis=0)
    rE, rM = _numpy_observables(dim, L, s, J)
    np.testing.assert_array_equal(E.cpu().numpy(), rE)
    np.testing.assert_array_equal(M.cpu().numpy(), rM)
    only = device_i32(I * R) + 1
    gbmc.observables(ctx, lat, None, only)
    np.testing.assert_array_equal(only.cpu().numpy(), rM)
    gbmc.lattice_free(lat)


@pytest.mark.parametrize("L,R", [(64, 5), (128, 1), (448, 3), (2048, 1)])
def test_bitpack_observables_and_conversion(ctx, L, R):
    lat = gbmc.lattice_init(ctx, 2, L, n_replicas=R, seed=3, layout=BP)
    E, M = device_i32(R) + 7, device_i32(R) - 3
    gbmc.observables(ctx, lat, E, M)
    s = spins_out(ctx, lat)
    np.testing.assert_array_equal(s[R - 1], oracle.init_spins(2, L, 3, 0, R - 1, True))
    rE, rM = _numpy_observables(2, L, s, None)
    np.testing.assert_array_equal(E.cpu().numpy(), rE)
    np.testing.assert_array_equal(M.cpu().numpy(), rM)
    # device buffers on any byte: written and read back
    buf = torch.zeros(R * L * L + 16, dtype=torch.int8, device="cuda")
    for off in (0, 1, 4, 10):
        view = buf[off:off + R * L * L]
        gbmc.lattice_copy_out(ctx, lat, view)
        np.testing.assert_array_equal(view.cpu().numpy().reshape(R, -1), s)
        flipped = (-s).reshape(-1)
        view.copy_(torch.from_numpy(flipped))
        gbmc.lattice_copy_in(ctx, lat, view)
        np.testing.assert_array_equal(spins_out(ctx, lat), -s)
        gbmc.lattice_copy_in(ctx, lat, np.ascontiguousarray(s))
    gbmc.lattice_free(lat)
