"""Which kernel sweeps many large copies: the bit-plane strips give a copy whole multiprocessors,
so copies that do not divide the device take the halo tiles where there are any, with the
oracle's configurations either way."""
import numpy as np
import pytest

import oracle
from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,halves,extra,series,kind", [
    (512, 1, 1, False, "sweep_tiles"),     # one block each on half of the device
    (512, 1, 0, False, "stream_strips"),   # two blocks each on all of it
    (512, 2, 1, False, "sweep_tiles"),     # a batch of one copy after a full one
    (512, 2, 0, False, "stream_strips"),
    (512, 1, 1, True, "stream_strips"),    # E and M after every sweep
    (486, 1, 1, False, "stream_strips"),   # no tiles of this size
])
def test_copies_that_do_not_divide_the_device(ctx, L, halves, extra, series, kind):
    R = halves * (torch.cuda.get_device_properties(0).multi_processor_count // 2) + extra
    lat = gbmc.lattice_init(ctx, 2, L, n_replicas=R, seed=41)
    E = device_i32(3 * R) if series else None
    gbmc.gbmc_profile(ctx, True)
    gbmc.metropolis_sweeps(ctx, lat, 0.44, 3, E, None)
    prof = gbmc.gbmc_profile_read(ctx)
    gbmc.gbmc_profile(ctx, False)
    assert kind in prof and not {"sweep_tiles", "stream_strips", "halfsweep_global"} & (set(prof) - {kind}), prof
    got = spins_out(ctx, lat)
    for c in (0, R // 2, R - 1):
        s = oracle.init_spins(2, L, 41, 0, c, True)
        oracle.sweeps(2, L, s, None, 0.44, 41, 0, c, 0, 3)
        np.testing.assert_array_equal(got[c], s)
        if series:
            assert E.cpu().numpy().reshape(3, R)[-1, c] == oracle.observables(2, L, s, None)[0]
    gbmc.lattice_free(lat)
