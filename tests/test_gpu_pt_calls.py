"""Rounds of tempering one, a few and many per call: a call of few rounds takes a sweep and an exchange
launch each where one launch for all would not pay, and so do instances whose clusters do not all
find room at once; the oracle's configurations and maps whatever the calls."""
import numpy as np
import pytest

import oracle
from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu
FM, EA = gbmc.GBMC_ISING_FM, gbmc.GBMC_EA_PMJ


@pytest.mark.parametrize("dim,L,model,I,T,theta,calls", [
    # (rounds of a call, whether they are one launch)
    (3, 8, EA, 2000, 4, 1, [(1, False), (20, True), (1, False), (5, True)]),
    (3, 8, EA, 1, 16, 2, [(1, True), (3, True)]),
    (2, 8, FM, 2000, 4, 1, [(20, True), (1, False)]),
    (3, 32, FM, 16, 16, 10, [(1, False), (4, False)]),
])
def test_calls(ctx, dim, L, model, I, T, theta, calls):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the line is for 152 multiprocessors")
    betas = np.linspace(0.2, 0.9, T)
    lat = gbmc.lattice_init(ctx, dim, L, model=model, n_instances=I, n_replicas=T, seed=91)
    pt = gbmc.pt_create(ctx, lat, betas, theta)
    for n, together in calls:
        gbmc.gbmc_profile(ctx, True)
        gbmc.pt_step(ctx, pt, n)
        prof = gbmc.gbmc_profile_read(ctx)
        gbmc.gbmc_profile(ctx, False)
        assert ("pt_rounds" in prof) == together and ("pt_exchange" in prof) != together, (n, prof)
    rep, E = np.empty(I * T, dtype=np.uint32), np.empty(I * T, dtype=np.int32)
    gbmc.pt_state_out(ctx, pt, rep, None, E)
    gbmc.pt_free(pt)
    got = spins_out(ctx, lat).reshape(I, T, -1)
    for i in sorted({0, I // 2, I - 1}) if L < 32 else [I - 1]:
        s, r, _, e = oracle.pt_run(dim, L, 91, i, betas, theta, sum(n for n, _ in calls),
                                   J=oracle.couplings(L, 91, i) if model == EA else None)
        np.testing.assert_array_equal(got[i], s)
        np.testing.assert_array_equal(rep.reshape(I, T)[i], r)
        np.testing.assert_array_equal(E.reshape(I, T)[i], e)
    gbmc.lattice_free(lat)
