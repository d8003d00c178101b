"""GPU parity of the sweeps that hold a large lattice's bit planes in global memory and
run every half-sweep of a call in one cooperative launch: against the CPU oracle on
sizes whose rows, slabs and planes end inside words, with runs of a few words per
thread block (four threads per word, several neighbours to wait for) and of many,
several copies, more copies than multiprocessors, E and M after every sweep, and the
bounded waits run out on purpose."""
import numpy as np
import pytest

import oracle
from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu

FM, EA, INT8, BP = gbmc.GBMC_ISING_FM, gbmc.GBMC_EA_PMJ, gbmc.GBMC_INT8, gbmc.GBMC_BITPACK


@pytest.mark.parametrize("dim,L,model,layout,I,R,beta,n", [
    (2, 258, FM, INT8, 1, 1, 0.44, 5),    # fits a block's shared memory, but alone
    (2, 284, FM, INT8, 1, 3, 0.44, 4),
    (2, 490, FM, INT8, 1, 2, 0.3, 3),
    (2, 512, FM, INT8, 2, 1, 0.44, 2),
    (2, 520, FM, INT8, 1, 1, 0.0, 2),     # beta = 0: every site flips
    (2, 666, FM, INT8, 1, 1, 20.0, 3),    # only dE <= 0 moves
    (2, 1000, FM, INT8, 1, 1, 0.44, 2),
    (2, 128, FM, INT8, 1, 1, 0.44, 8),
    (2, 486, FM, INT8, 1, 170, 0.44, 2),  # more copies than multiprocessors
    (2, 64, FM, BP, 1, 2, 0.44, 4),
    (2, 448, FM, BP, 3, 1, 0.44, 3),
    (2, 1024, FM, BP, 1, 1, 0.44, 2),
    (3, 32, EA, INT8, 1, 2, 1.1, 8),
    (3, 34, FM, INT8, 1, 1, 0.22, 4),
    (3, 40, EA, INT8, 2, 1, 1.1, 3),
    (3, 42, EA, INT8, 1, 2, 1.1, 2),
    (3, 62, FM, INT8, 1, 1, 0.22, 2),
    (3, 66, EA, INT8, 1, 1, 0.0, 2),
])
def test_stream_strips_match_oracle(ctx, dim, L, model, layout, I, R, beta, n):
    seed, C = 100 + L, I * R
    lat = gbmc.lattice_init(ctx, dim, L, model=model, n_instances=I, n_replicas=R, seed=seed, instance_base=4,
                            layout=layout)
    gbmc.lattice_set_sweep_counter(lat, 7)
    Es, Ms = device_i32(n * C) + 5, device_i32(n * C) - 5
    gbmc.gbmc_profile(ctx, True)
    gbmc.metropolis_sweeps(ctx, lat, beta, n, Es, Ms)
    prof = gbmc.gbmc_profile_read(ctx)
    gbmc.gbmc_profile(ctx, False)
    assert "stream_strips" in prof and "halfsweep_global" not in prof and "observables" not in prof
    got = spins_out(ctx, lat)
    Es, Ms = Es.cpu().numpy().reshape(n, C), Ms.cpu().numpy().reshape(n, C)
    for c in range(C) if C <= 4 else (0, 1, C // 2, 151, 152, C - 1):
        i, r = divmod(c, R)
        J = oracle.couplings(L, seed, 4 + i) if model == EA else None
        s = oracle.init_spins(dim, L, seed, 4 + i, r, True)
        for t in range(n):
            oracle.sweeps(dim, L, s, J, beta, seed, 4 + i, r, 7 + t, 1)
            assert (Es[t, c], Ms[t, c]) == oracle.observables(dim, L, s, J), (c, t)
        np.testing.assert_array_equal(got[c], s)
    # without series, counters continued
    gbmc.metropolis_sweeps(ctx, lat, beta, 4)
    i, r = divmod(C - 1, R)
    oracle.sweeps(dim, L, s, J, beta, seed, 4 + i, r, 7 + n, 4)
    np.testing.assert_array_equal(spins_out(ctx, lat)[C - 1], s)
    gbmc.lattice_free(lat)


def test_stream_strips_equal_byte_kernels_over_many_sweeps(ctx):
    # 400 half-sweeps of exchanged words; energies at every sweep
    for dim, L, model in ((2, 1000, FM), (2, 330, FM), (3, 48, EA)):
        out = []
        for kernel in (gbmc.GBMC_KERNEL_AUTO, gbmc.GBMC_KERNEL_BYTES):
            gbmc.gbmc_set_sweep_kernel(ctx, kernel)
            lat = gbmc.lattice_init(ctx, dim, L, model=model, seed=9)
            E, M = device_i32(200), device_i32(200)
            gbmc.metropolis_sweeps(ctx, lat, 0.44 if dim == 2 else 0.9, 200, E, M)
            out.append((spins_out(ctx, lat), E.cpu().numpy(), M.cpu().numpy()))
            gbmc.lattice_free(lat)
        gbmc.gbmc_set_sweep_kernel(ctx, gbmc.GBMC_KERNEL_AUTO)
        for a, b in zip(out[0], out[1]):
            np.testing.assert_array_equal(a, b)


def test_stream_strips_wait_runs_out_and_is_reported(ctx):
    lat = gbmc.lattice_init(ctx, 2, 520, seed=6)
    gbmc.gbmc_test_barrier_wait(ctx, 1, 2_000_000)  # ~1 ms budget, one phantom half-sweep
    try:
        gbmc.metropolis_sweeps(ctx, lat, 0.44, 4)
        with pytest.raises(gbmc.GbmcError) as e:
            gbmc.gbmc_sync(ctx)
        assert e.value.status == gbmc.GBMC_ERR_TIMEOUT
    finally:
        gbmc.gbmc_test_barrier_wait(ctx, 0, 2_000_000_000)
    gbmc.gbmc_sync(ctx)
    gbmc.lattice_free(lat)
    lat = gbmc.lattice_init(ctx, 2, 520, seed=6)
    gbmc.metropolis_sweeps(ctx, lat, 0.44, 4)
    s = oracle.init_spins(2, 520, 6, 0, 0, True)
    oracle.sweeps(2, 520, s, None, 0.44, 6, 0, 0, 0, 4)
    np.testing.assert_array_equal(spins_out(ctx, lat)[0], s)
    gbmc.lattice_free(lat)
