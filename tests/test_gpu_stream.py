"""GPU parity of the bit-stream resident sweep kernel (any even L, several copies
per thread): against the CPU oracle element by element on sizes whose rows,
slabs and planes end inside words, and against the byte-plane kernel on
populations large enough for two and four copies per thread and for whole-block
teams, with copy counts that leave groups, warps and blocks partly empty."""
import numpy as np
import pytest

import oracle
from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, spins_out, torch  # noqa: F401
from tests.test_gpu_pa import _compare_run

pytestmark = pytest.mark.gpu

FM, EA = gbmc.GBMC_ISING_FM, gbmc.GBMC_EA_PMJ


def _kinds(ctx, fn):
    gbmc.gbmc_profile(ctx, True)
    fn()
    prof = gbmc.gbmc_profile_read(ctx)
    gbmc.gbmc_profile(ctx, False)
    return prof


@pytest.mark.parametrize("dim,L,model,I,R,beta,n", [
    (2, 2, FM, 1, 3, 0.4, 4),       # a plane of 2 sites
    (2, 4, FM, 2, 5, 0.44, 4),
    (2, 6, FM, 1, 7, 0.3, 4),
    (2, 10, FM, 1, 9, 0.44, 4),
    (2, 18, FM, 2, 5, 0.5, 3),
    (2, 24, FM, 1, 3, 0.0, 2),      # beta = 0: every site flips
    (2, 40, FM, 1, 2, 20.0, 3),     # only dE <= 0 moves
    (2, 66, FM, 1, 3, 0.44, 3),
    (2, 96, FM, 1, 2, 0.44, 3),
    (2, 200, FM, 1, 2, 0.44, 2),
    (2, 320, FM, 1, 1, 0.44, 2),    # a whole block per copy
    (3, 2, EA, 3, 5, 0.8, 4),
    (3, 4, EA, 2, 9, 1.1, 4),       # a plane of one whole word
    (3, 6, EA, 3, 7, 1.1, 4),
    (3, 10, EA, 2, 5, 1.1, 3),
    (3, 12, FM, 1, 5, 0.22, 3),
    (3, 14, EA, 1, 3, 0.0, 2),
    (3, 20, EA, 2, 2, 1.1, 2),
    (3, 32, EA, 1, 2, 1.1, 2),
    (3, 38, FM, 1, 2, 0.22, 1),
    # populations too small for the kernel of the fixed sizes
    (2, 16, FM, 2, 5, 0.44, 3),
    (2, 32, FM, 1, 7, 0.44, 3),
    (2, 64, FM, 1, 3, 0.44, 3),
    (2, 128, FM, 1, 2, 0.44, 2),
    (2, 256, FM, 1, 1, 0.44, 2),
    (3, 8, EA, 2, 3, 1.1, 3),
    (3, 16, EA, 1, 2, 1.1, 2),
])
def test_stream_sweeps_match_oracle(ctx, dim, L, model, I, R, beta, n):
    seed, C = 1000 + 10 * L + dim, I * R
    lat = gbmc.lattice_init(ctx, dim, L, model=model, n_instances=I, n_replicas=R, seed=seed, instance_base=4,
                            start=gbmc.GBMC_START_RANDOM)
    Es, Ms = device_i32(n * C), device_i32(n * C)
    prof = _kinds(ctx, lambda: gbmc.metropolis_sweeps(ctx, lat, beta, n, Es, Ms))
    assert "sweep_stream" in prof and "sweep_resident" not in prof
    got = spins_out(ctx, lat)
    Es, Ms = Es.cpu().numpy().reshape(n, C), Ms.cpu().numpy().reshape(n, C)
    for c in range(C):
        i, r = divmod(c, R)
        J = oracle.couplings(L, seed, 4 + i) if model == EA else None
        s = oracle.init_spins(dim, L, seed, 4 + i, r, True)
        for t in range(n):
            oracle.sweeps(dim, L, s, J, beta, seed, 4 + i, r, t, 1)
            assert (Es[t, c], Ms[t, c]) == oracle.observables(dim, L, s, J), (c, t)
        np.testing.assert_array_equal(got[c], s)
    gbmc.lattice_free(lat)


@pytest.mark.parametrize("dim,L,model,I,R", [
    (2, 8, FM, 1, 20011),     # a plane of one whole word
    (2, 12, FM, 1, 70001),    # four copies per thread, 3 words per plane
    (2, 24, FM, 1, 34603),
    (2, 24, FM, 1, 9001),     # two
    (2, 64, FM, 1, 500),      # one, a word per thread
    (2, 48, FM, 3, 2903),
    (2, 96, FM, 1, 2161),
    (2, 204, FM, 1, 481),     # whole-block teams
    (3, 4, EA, 7, 44491),
    (3, 6, EA, 5, 15561),
    (3, 10, EA, 3, 6603),
    (3, 10, FM, 1, 10001),
    (3, 12, EA, 3, 3847),
    (3, 24, EA, 2, 721),
    (3, 32, FM, 1, 307),
])
def test_stream_equals_bytes_kernel(ctx, dim, L, model, I, R):
    out = []
    for kernel in (gbmc.GBMC_KERNEL_AUTO, gbmc.GBMC_KERNEL_BYTES):
        gbmc.gbmc_set_sweep_kernel(ctx, kernel)
        lat = gbmc.lattice_init(ctx, dim, L, model=model, n_instances=I, n_replicas=R, seed=77,
                                start=gbmc.GBMC_START_RANDOM)
        E, M = device_i32(2 * I * R), device_i32(2 * I * R)
        prof = _kinds(ctx, lambda: gbmc.metropolis_sweeps(ctx, lat, 0.7 if dim == 3 else 0.44, 2, E, M))
        assert ("sweep_stream" in prof) == (kernel == gbmc.GBMC_KERNEL_AUTO)
        out.append((spins_out(ctx, lat), E.cpu().numpy(), M.cpu().numpy()))
        gbmc.lattice_free(lat)
    gbmc.gbmc_set_sweep_kernel(ctx, gbmc.GBMC_KERNEL_AUTO)
    for a, b in zip(out[0], out[1]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("law", [gbmc.GBMC_RESAMPLE_MULTINOMIAL, gbmc.GBMC_RESAMPLE_NEAREST])
def test_stream_annealing_matches_oracle(ctx, law):
    # gather through the parents, live slots only; a spin glass with three instances
    L, I, R0, cap, S, theta, seed = 6, 3, 150, 220, 5, 2, 9
    R = cap if law else R0
    lat = gbmc.lattice_init(ctx, 3, L, model=EA, n_instances=I, n_replicas=R, seed=seed, instance_base=10)
    betas = oracle.linear_betas(2.0, S)
    pa = gbmc.pa_create(ctx, [lat], theta, S, schedule=gbmc.GBMC_SCHED_LIST, betas=betas, resample=law,
                        initial_replicas=R0 if law else 0)
    stats, _ = gbmc.pa_run(ctx, pa, capacity=S + 1)
    got = spins_out(ctx, lat).reshape(I, R, -1)
    for i in range(I):
        J = oracle.couplings(L, seed, 10 + i)
        if law:
            ref = oracle.pa_run_nearest(3, L, seed, 10 + i, R0, cap, betas, theta, J=J)
            np.testing.assert_array_equal(stats[:, i]["n_replicas"], ref["nrep"])
            np.testing.assert_array_equal(stats[:, i]["sumE"], ref["sumE"])
        else:
            ref = oracle.pa_run(3, L, seed, 10 + i, R, betas, theta, J=J)
            _compare_run(stats, ref, i, L ** 3)
        np.testing.assert_array_equal(got[i][:len(ref["spins"])], ref["spins"])
    gbmc.pa_free(pa)
    gbmc.lattice_free(lat)


@pytest.mark.parametrize("L,I,T", [(6, 3, 9), (12, 2, 6)])
def test_stream_parallel_tempering_matches_oracle(ctx, L, I, T):
    theta, steps, seed = 3, 12, 41
    betas = np.linspace(0.2, 1.4, T)
    lat = gbmc.lattice_init(ctx, 3, L, model=EA, n_instances=I, n_replicas=T, seed=seed, instance_base=2)
    pt = gbmc.pt_create(ctx, lat, betas, theta)
    gbmc.pt_step(ctx, pt, steps)
    rep, E = np.empty(I * T, dtype=np.uint32), np.empty(I * T, dtype=np.int32)
    gbmc.pt_state_out(ctx, pt, rep, None, E)
    gbmc.pt_free(pt)
    got = spins_out(ctx, lat).reshape(I, T, -1)
    for i in range(I):
        s, r, _, e = oracle.pt_run(3, L, seed, 2 + i, betas, theta, steps, J=oracle.couplings(L, seed, 2 + i))
        np.testing.assert_array_equal(got[i], s)
        np.testing.assert_array_equal(rep.reshape(I, T)[i], r)
        np.testing.assert_array_equal(E.reshape(I, T)[i], e)
    gbmc.lattice_free(lat)
