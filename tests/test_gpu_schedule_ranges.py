"""Adaptive steps by bisection over histograms of every width the kernel treats
differently: one level (the largest step is taken), a few bins, several bins per
thread, the widest range kept on chip and one beyond it. The chosen step against the
oracle's sequential bisection: both halve the same interval 50 times, so they
differ by what the overlap's rounding (1e-14) moves its crossing of the target, a
relative 1e-13 of a step, and by the last interval, 0.1 x 2^-50 against steps of 1e-6
and more: 1e-9 holds with room."""
import numpy as np
import pytest

from oracle import schedule as osch
from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, torch  # noqa: F401

pytestmark = pytest.mark.gpu


# (L, copies, bins between the ground state and a random copy: about L^2 / 2)
@pytest.mark.parametrize("L,R", [(16, 1), (16, 5), (48, 300), (88, 200), (96, 200), (128, 40)])
def test_bisection_over_wide_histograms(ctx, L, R):
    rng = np.random.default_rng(L + R)
    spins = np.ones((R, L * L), dtype=np.int8)
    for r in range(1, R):  # from the ground state to half of the spins turned
        flip = rng.random(L * L) < 0.5 * r / (R - 1)
        spins[r, flip] = -1
    lat = gbmc.lattice_init(ctx, 2, L, n_replicas=R, seed=3)
    gbmc.lattice_copy_in(ctx, lat, spins)
    pa = gbmc.pa_create(ctx, [lat], 1, 400, schedule=gbmc.GBMC_SCHED_BISECTION, beta_f=1.0, init=False,
                        target_overlap=0.85, dbeta_max=0.1)
    E = np.empty(R, dtype=np.int32)
    gbmc.pa_energies_out(ctx, pa, 0, E)
    assert R == 1 or int(E.max()) - int(E.min()) >= 1.5 * L * L
    gbmc.pa_step(ctx, pa)
    rec = gbmc.pa_schedule_log(pa, 0)[0]
    levels, counts = osch.histogram(E.astype(np.int64))
    ch = osch.choose_step(levels, counts, 0.0, L, R, L * L, 0.1, 0.85)
    assert rec["kind"] == 1 and rec["evals"] == ch["evals"]
    assert rec["dbeta"] == pytest.approx(ch["dbeta"], rel=1e-9)
    assert rec["alpha"] == pytest.approx(ch["alpha"], rel=1e-9)
    assert bool(rec["clamped"]) == (R == 1)
    f = osch.features(levels, counts, 0.0, L, R, L * L)
    np.testing.assert_allclose(rec["features"], f.astype(np.float32), rtol=1e-6, atol=1e-6)
    gbmc.pa_free(pa)
    gbmc.lattice_free(lat)
