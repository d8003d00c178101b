"""The bounds-checked build over the kernels that the default (AUTO) mode takes: sweeps with bits
drawn ahead and bit-stream sweeps on both sides of the multiprocessor count, large lattices in
bit-plane strips (runs of a few words, many, and held in shared memory, several copies, E and M),
Swendsen-Wang on chip, in tiles cut by the lattice's edge and untiled, resampling in clusters and
above their limits, adaptive steps, rounds of tempering. No check may fail (gbmc_sync reports one)
and the oracle's configurations come out. It runs in a child process that loads the checked library."""
import os
import subprocess
import sys

import pytest

from paper_1709_04394_gb300 import build as gbuild
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = r'''
import numpy as np, torch
import oracle
from paper_1709_04394_gb300 import gbmc
assert gbmc.gbmc_checked_build()
ctx = gbmc.gbmc_create(0, torch.cuda.current_stream().cuda_stream)
FM, EA, INT8, BP = gbmc.GBMC_ISING_FM, gbmc.GBMC_EA_PMJ, gbmc.GBMC_INT8, gbmc.GBMC_BITPACK
SMS = torch.cuda.get_device_properties(0).multi_processor_count
i32 = lambda n: torch.zeros(n, dtype=torch.int32, device="cuda")

def spins(lat):
    info = gbmc.lattice_info(lat)
    h = np.empty((info.n_copies, info.n_sites), dtype=np.int8)
    gbmc.lattice_copy_out(ctx, lat, h)
    return h

def kinds(fn):
    gbmc.gbmc_profile(ctx, True)
    fn()
    gbmc.gbmc_sync(ctx)
    prof = gbmc.gbmc_profile_read(ctx)
    gbmc.gbmc_profile(ctx, False)
    return prof
'''

SWEEPS = HEAD + r'''
for kind, cases in (
    ("sweep_stream", [(2, 2, FM, INT8, 3), (2, 4, FM, INT8, 2), (2, 6, FM, INT8, SMS + 1), (2, 16, FM, INT8, 1), (2, 18, FM, INT8, 3),
                      (2, 44, FM, INT8, 2), (2, 46, FM, INT8, 2), (2, 90, FM, INT8, 2), (2, 24, FM, INT8, SMS + 1),
                      (2, 66, FM, INT8, SMS + 3), (2, 204, FM, INT8, SMS + 1), (2, 12, FM, INT8, 70001), (2, 96, FM, INT8, 2161),
                      (3, 2, EA, INT8, 3), (3, 4, EA, INT8, 5), (3, 10, EA, INT8, 3), (3, 20, FM, INT8, 2),
                      (3, 10, EA, INT8, SMS + 5), (3, 6, EA, INT8, 40000)]),
    ("stream_strips", [(2, 258, FM, INT8, 1), (2, 490, FM, INT8, 3), (2, 760, FM, INT8, 1), (2, 1000, FM, INT8, 1),
                       (2, 486, FM, INT8, SMS + 1), (2, 64, FM, BP, 2), (2, 448, FM, BP, 3), (3, 34, FM, INT8, 1),
                       (3, 32, EA, INT8, 2), (3, 62, FM, INT8, 1), (3, 66, EA, INT8, 1), (3, 40, EA, INT8, 9)])):
    for dim, L, model, layout, R in cases:
        lat = gbmc.lattice_init(ctx, dim, L, model=model, n_replicas=R, seed=3, instance_base=1, layout=layout)
        n, m = (3, 2) if kind == "sweep_stream" else (8, 8)
        E, M = i32(n * R), i32(n * R)
        prof = kinds(lambda: (gbmc.metropolis_sweeps(ctx, lat, 0.4, n, E, M), gbmc.metropolis_sweeps(ctx, lat, 0.7, m)))
        assert kind in prof and "sweep_resident" not in prof and "halfsweep_global" not in prof, (L, prof)
        c = R - 1
        J = oracle.couplings(L, 3, 1) if model == EA else None
        s = oracle.init_spins(dim, L, 3, 1, c, True)
        oracle.sweeps(dim, L, s, J, 0.4, 3, 1, c, 0, n)
        assert (E.view(n, R)[n - 1, c].item(), M.view(n, R)[n - 1, c].item()) == oracle.observables(dim, L, s, J)
        oracle.sweeps(dim, L, s, J, 0.7, 3, 1, c, n, m)
        assert np.array_equal(spins(lat)[c], s), (dim, L, model, R)
        gbmc.lattice_free(lat)
print("checked ok")
'''

OTHERS = HEAD + r'''
# Swendsen-Wang: 2D L = 2 and 3D L = 34 take the untiled kernels, small lattices stay on chip, L = 34 and 66 have cut tiles
for dim, L, R in [(2, 2, 3), (2, 4, 3), (2, 6, 2), (2, 34, 3), (2, 66, 2), (2, 100, SMS + 1), (2, 130, 2), (2, 192, 1),
                  (3, 4, 3), (3, 6, 2), (3, 8, 3), (3, 10, 1), (3, 34, 1), (3, 32, 1)]:
    lat = gbmc.lattice_init(ctx, dim, L, n_replicas=R, seed=9)
    E, M = i32(3 * R), i32(3 * R)
    gbmc.swendsen_wang(ctx, lat, 0.4, 3, E, M)
    gbmc.swendsen_wang(ctx, lat, 0.3, 1)
    gbmc.gbmc_sync(ctx)
    s = oracle.init_spins(dim, L, 9, 0, R - 1, True)
    for t in range(3):
        oracle.sw_update(dim, L, s, 0.4, 9, 0, R - 1, t)
    assert (E.view(3, R)[2, R - 1].item(), M.view(3, R)[2, R - 1].item()) == oracle.observables(dim, L, s, None)
    oracle.sw_update(dim, L, s, 0.3, 9, 0, R - 1, 3)
    assert np.array_equal(spins(lat)[R - 1], s), (dim, L)
    gbmc.lattice_free(lat)
# resampling: slices of 7 and 15 workers, many populations, populations beyond the clusters
for law, R, I in [(0, 37, 3), (0, 2049, 1), (0, 7681, 1), (0, 24577, 1), (0, 20, 150), (1, 61, 2), (1, 4001, 1), (1, 65537, 1),
                  (2, 61, 2), (2, 4001, 1), (2, 8193, 1)]:
    lat = gbmc.lattice_init(ctx, 3, 4, model=EA, n_instances=I, n_replicas=R, seed=6)
    pa = gbmc.pa_create(ctx, [lat], 1, 3, beta_f=0.6, resample=law, initial_replicas=R * 3 // 4 if law and R > 100 else 31 if law else 0)
    gbmc.pa_run(ctx, pa, capacity=4)
    gbmc.gbmc_sync(ctx)
    gbmc.pa_free(pa)
    gbmc.lattice_free(lat)
# adaptive steps
for L, R in [(6, 200), (64, 300), (128, 40)]:
    lat = gbmc.lattice_init(ctx, 2, L, n_replicas=R, seed=7)
    pa = gbmc.pa_create(ctx, [lat], 1, 4096, schedule=gbmc.GBMC_SCHED_BISECTION, beta_f=0.05, target_overlap=0.85)
    gbmc.pa_run(ctx, pa, capacity=4097)
    gbmc.gbmc_sync(ctx)
    gbmc.pa_free(pa)
    gbmc.lattice_free(lat)
# tempering in rounds and a launch per round
for L, I, T in [(4, 3, 5), (8, 2, 9), (10, 3, 7), (8, 400, 8)]:
    lat = gbmc.lattice_init(ctx, 3, L, model=EA, n_instances=I, n_replicas=T, seed=8)
    pt = gbmc.pt_create(ctx, lat, np.linspace(0.2, 1.0, T), 2)
    gbmc.pt_step(ctx, pt, 4)
    gbmc.gbmc_sync(ctx)
    gbmc.pt_free(pt)
    got = spins(lat)
    s, _, _, _ = oracle.pt_run(3, L, 8, I - 1, np.linspace(0.2, 1.0, T), 2, 4, J=oracle.couplings(L, 8, I - 1))
    assert np.array_equal(got.reshape(I, T, -1)[I - 1], s), (L, I, T)
    gbmc.lattice_free(lat)
print("checked ok")
'''


@pytest.mark.parametrize("script", [SWEEPS, OTHERS], ids=["sweeps", "others"])
def test_default_kernels_record_no_bounds_failure(script):
    require_gpu()
    gbuild.build(check=True)
    env = dict(os.environ, GBMC_LIBRARY="libgbmc_check.so")
    r = subprocess.run([sys.executable, "-c", script], cwd=ROOT, env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "checked ok" in r.stdout
