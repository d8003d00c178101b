"""Calls whose faster kernels want a buffer that cannot be had -- the allocator refuses it, or
the stream is being captured -- take the kernels that need none, with the same results."""
import numpy as np
import pytest

import oracle
from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, require_gpu, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu
FM, EA, INT8, BP = gbmc.GBMC_ISING_FM, gbmc.GBMC_EA_PMJ, gbmc.GBMC_INT8, gbmc.GBMC_BITPACK
N_SWEEPS = 4


def _sweep(dim, L, model, seed, c, beta, t0):
    """The oracle's copy c after N_SWEEPS sweeps from t0 on, and E, M after each."""
    J = oracle.couplings(L, seed, 0) if model == EA else None
    s = oracle.init_spins(dim, L, seed, 0, c, True)
    EM = []
    for t in range(t0 + N_SWEEPS):
        oracle.sweeps(dim, L, s, J, beta, seed, 0, c, t, 1)
        EM.append(oracle.observables(dim, L, s, J))
    return s, EM[t0:]


@pytest.mark.parametrize("dim,L,model,layout,R", [
    (2, 500, FM, INT8, 2), (2, 512, FM, INT8, 1), (2, 448, FM, BP, 2), (3, 62, FM, INT8, 1), (3, 40, EA, INT8, 2)])
def test_large_lattices_without_the_buffer(ctx, dim, L, model, layout, R):
    lat = gbmc.lattice_init(ctx, dim, L, model=model, n_replicas=R, seed=31, layout=layout)
    E, M = device_i32(N_SWEEPS * R), device_i32(N_SWEEPS * R)
    for t0, limit in ((0, 1000), (N_SWEEPS, 2**64 - 1)):
        gbmc.gbmc_test_spare_limit(ctx, limit)
        gbmc.gbmc_profile(ctx, True)
        try:
            gbmc.metropolis_sweeps(ctx, lat, 0.4, N_SWEEPS, E, M)
        finally:
            gbmc.gbmc_test_spare_limit(ctx)
        prof = gbmc.gbmc_profile_read(ctx)
        gbmc.gbmc_profile(ctx, False)
        assert ("stream_strips" in prof) == (t0 > 0), prof
        s, EM = _sweep(dim, L, model, 31, R - 1, 0.4, t0)
        np.testing.assert_array_equal(spins_out(ctx, lat)[R - 1], s)
        np.testing.assert_array_equal(E.cpu().numpy().reshape(N_SWEEPS, R)[:, -1], [e for e, _ in EM])
        np.testing.assert_array_equal(M.cpu().numpy().reshape(N_SWEEPS, R)[:, -1], [m for _, m in EM])
    gbmc.lattice_free(lat)


@pytest.mark.parametrize("dim,L,model", [(2, 12, FM), (3, 6, EA), (3, 40, EA)])
def test_lattices_without_bit_stream_tables(ctx, dim, L, model):
    gbmc.gbmc_test_spare_limit(ctx, 0)
    try:
        lat = gbmc.lattice_init(ctx, dim, L, model=model, n_replicas=3, seed=32)
    finally:
        gbmc.gbmc_test_spare_limit(ctx)
    gbmc.gbmc_profile(ctx, True)
    gbmc.metropolis_sweeps(ctx, lat, 0.4, N_SWEEPS)
    prof = gbmc.gbmc_profile_read(ctx)
    gbmc.gbmc_profile(ctx, False)
    assert "sweep_stream" not in prof and "stream_strips" not in prof
    np.testing.assert_array_equal(spins_out(ctx, lat)[2], _sweep(dim, L, model, 32, 2, 0.4, 0)[0])
    if L == 6:  # tempering, annealing
        pt = gbmc.pt_create(ctx, lat, np.linspace(0.3, 0.9, 3), 2)
        gbmc.pt_step(ctx, pt, 3)
        gbmc.pt_free(pt)
        pa = gbmc.pa_create(ctx, [lat], 2, 3, beta_f=0.5)
        gbmc.pa_run(ctx, pa, capacity=4)
        gbmc.pa_free(pa)
    gbmc.lattice_free(lat)


@pytest.mark.parametrize("dim,L,layout,series", [(2, 500, INT8, False), (3, 62, INT8, True), (2, 448, BP, True)])
def test_first_call_of_a_large_lattice_can_be_captured(dim, L, layout, series):
    require_gpu()
    stream = torch.cuda.Stream()
    own = gbmc.gbmc_create(0, stream.cuda_stream)
    E, M = (device_i32(N_SWEEPS), device_i32(N_SWEEPS)) if series else (None, None)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        lat = gbmc.lattice_init(own, dim, L, seed=33, layout=layout)
        warm = gbmc.lattice_init(own, dim, L, seed=34, layout=layout)  # the kernels loaded before the capture
        gbmc.gbmc_set_sweep_launch(own, gbmc.GBMC_LAUNCH_GRID)
        gbmc.metropolis_sweeps(own, warm, 0.4, N_SWEEPS, E, M)
        gbmc.gbmc_set_sweep_launch(own, gbmc.GBMC_LAUNCH_AUTO)
        gbmc.gbmc_sync(own)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            gbmc.metropolis_sweeps(own, lat, 0.4, N_SWEEPS, E, M)
        graph.replay()
        gbmc.gbmc_sync(own)
        s, EM = _sweep(dim, L, FM, 33, 0, 0.4, 0)
        np.testing.assert_array_equal(spins_out(own, lat)[0], s)
        if series:
            np.testing.assert_array_equal(E.cpu().numpy(), [e for e, _ in EM])
            np.testing.assert_array_equal(M.cpu().numpy(), [m for _, m in EM])
        # the next call is not captured and goes on from there
        gbmc.metropolis_sweeps(own, lat, 0.4, N_SWEEPS)
        s, _ = _sweep(dim, L, FM, 33, 0, 0.4, N_SWEEPS)
        np.testing.assert_array_equal(spins_out(own, lat)[0], s)
    gbmc.lattice_free(lat)
    gbmc.lattice_free(warm)
    gbmc.gbmc_destroy(own)
