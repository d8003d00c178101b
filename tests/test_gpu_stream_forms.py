"""Every form of the bit-stream kernel (four, two or one copy per thread, two or four threads per
word, one-warp and whole-block teams) against the CPU oracle, with E and M after every sweep, on
more copies than multiprocessors: fewer have their bits drawn ahead by another kernel. The
form a case means to run is asserted; sizes whose planes are a part of a word, end inside a word or
on its edge; copy counts that leave groups and teams partly empty."""
import numpy as np
import pytest

import oracle
from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu
FM, EA = gbmc.GBMC_ISING_FM, gbmc.GBMC_EA_PMJ
WARP, BLOCK = "one-warp teams", "a block per team"


@pytest.mark.parametrize("dim,L,model,I,R,beta,copies,threads,team", [
    # a quarter of a word per thread
    (2, 2, FM, 1, 201, 0.4, 1, 4, WARP),      # a plane of 2 sites
    (2, 4, FM, 3, 67, 0.44, 1, 4, WARP),
    (2, 6, FM, 1, 203, 0.3, 1, 4, WARP),
    (2, 10, FM, 1, 201, 0.44, 1, 4, WARP),
    (2, 18, FM, 2, 101, 0.5, 1, 4, WARP),
    (2, 24, FM, 1, 201, 0.0, 1, 4, BLOCK),    # beta = 0: every site flips
    (2, 40, FM, 1, 201, 20.0, 1, 4, BLOCK),   # only dE <= 0 moves
    (3, 2, EA, 3, 71, 0.8, 1, 4, WARP),
    (3, 4, EA, 2, 101, 1.1, 1, 4, WARP),      # a plane of one whole word
    (3, 6, EA, 3, 67, 1.1, 1, 4, WARP),
    (3, 10, EA, 2, 101, 1.1, 1, 4, BLOCK),
    (3, 12, FM, 1, 201, 0.22, 1, 4, BLOCK),
    # half a word
    (2, 8, FM, 1, 20011, 0.44, 1, 2, WARP),
    (2, 24, FM, 1, 1513, 0.44, 1, 2, WARP),
    (2, 66, FM, 1, 201, 0.44, 1, 2, BLOCK),
    (3, 6, EA, 3, 1345, 0.9, 1, 2, WARP),
    (3, 14, EA, 1, 201, 0.0, 1, 2, BLOCK),
    # a word
    (2, 24, FM, 1, 9001, 0.44, 1, 1, WARP),
    (2, 204, FM, 1, 201, 0.44, 1, 1, BLOCK),
    (3, 10, FM, 1, 10001, 0.22, 1, 1, WARP),
    (3, 20, EA, 2, 81, 1.1, 1, 1, BLOCK),
    # two copies' words
    (2, 96, FM, 1, 2161, 0.44, 2, 1, BLOCK),
    (3, 4, EA, 7, 44491, 1.1, 2, 1, WARP),
    (3, 24, EA, 2, 721, 0.9, 2, 1, BLOCK),
    # four
    (2, 12, FM, 1, 70001, 0.44, 4, 1, WARP),
    (2, 24, FM, 1, 34603, 20.0, 4, 1, WARP),
    (2, 66, FM, 1, 2002, 0.44, 4, 1, BLOCK),
    (3, 6, EA, 5, 15561, 0.0, 4, 1, WARP),
    (3, 10, EA, 3, 6603, 1.1, 4, 1, WARP),
])
def test_forms_match_oracle(ctx, dim, L, model, I, R, beta, copies, threads, team):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert I * R > sms  # not the kernel of few copies
    f = gbmc.gbmc_test_stream_form([(dim, L, I, R)], sm_count=sms)
    if sms == 152:
        assert (f.copies_per_thread, f.threads_per_word) == (copies, threads)
        assert (team == WARP) == (f.team[0] == 32)
    seed, C, n = 500 + 10 * L + dim, I * R, 3
    lat = gbmc.lattice_init(ctx, dim, L, model=model, n_instances=I, n_replicas=R, seed=seed, instance_base=4)
    gbmc.lattice_set_sweep_counter(lat, 5)
    Es, Ms = device_i32(n * C), device_i32(n * C)
    # (the sums of 2D L = 8 with a series are the byte-plane kernel's up to 10 000 copies)
    gbmc.gbmc_profile(ctx, True)
    gbmc.metropolis_sweeps(ctx, lat, beta, n, Es, Ms)
    prof = gbmc.gbmc_profile_read(ctx)
    gbmc.gbmc_profile(ctx, False)
    assert list(prof) == ["sweep_stream"], prof
    got = spins_out(ctx, lat)
    Es, Ms = Es.cpu().numpy().reshape(n, C), Ms.cpu().numpy().reshape(n, C)
    for c in sorted({0, 1, R - 1, C // 2, C - 2, C - 1}):
        i, r = divmod(c, R)
        J = oracle.couplings(L, seed, 4 + i) if model == EA else None
        s = oracle.init_spins(dim, L, seed, 4 + i, r, True)
        for t in range(n):
            oracle.sweeps(dim, L, s, J, beta, seed, 4 + i, r, 5 + t, 1)
            assert (Es[t, c], Ms[t, c]) == oracle.observables(dim, L, s, J), (c, t)
        np.testing.assert_array_equal(got[c], s)
    gbmc.lattice_free(lat)
