"""Sweeps of few small copies, whose acceptance bits other warps draw ahead, against the
byte-plane kernel (the general path): configurations, E and M after every sweep, word for word.
Sizes: one word per plane and parts of one, planes that end inside a word, the most words
that one and that several updating warps take, the largest lattice and the next; sweeps: the fewest,
and enough for the ring of drawn words to come round many times; copies: as many as
multiprocessors, and one more (the other kernel)."""
import numpy as np
import pytest

from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, device_i32, spins_out, torch  # noqa: F401

pytestmark = pytest.mark.gpu
FM, EA = gbmc.GBMC_ISING_FM, gbmc.GBMC_EA_PMJ


def _run(ctx, kernel, dim, L, model, I, R, n, series):
    gbmc.gbmc_set_sweep_kernel(ctx, kernel)
    try:
        lat = gbmc.lattice_init(ctx, dim, L, model=model, n_instances=I, n_replicas=R, seed=50 + L, instance_base=2)
        gbmc.lattice_set_sweep_counter(lat, 9)
        E = device_i32(n * I * R) if "E" in series else None
        M = device_i32(n * I * R) if "M" in series else None
        gbmc.metropolis_sweeps(ctx, lat, 0.44 if dim == 2 else 0.3, n, E, M)
        gbmc.metropolis_sweeps(ctx, lat, 0.6, 2)  # the counter goes on
        gbmc.gbmc_sync(ctx)
        out = [spins_out(ctx, lat)] + [x.cpu().numpy() for x in (E, M) if x is not None]
        gbmc.lattice_free(lat)
        return out
    finally:
        gbmc.gbmc_set_sweep_kernel(ctx, gbmc.GBMC_KERNEL_AUTO)


@pytest.mark.parametrize("dim,L,model,I,R,n,series", [
    (2, 4, FM, 1, 2, 40, "EM"), (2, 6, FM, 1, 3, 40, "EM"), (2, 8, FM, 1, 5, 700, "EM"), (2, 10, FM, 1, 1, 40, "E"),
    (2, 16, FM, 1, 1, 2, "EM"), (2, 16, FM, 1, 1, 1500, "EM"), (2, 44, FM, 1, 2, 60, "EM"), (2, 46, FM, 1, 2, 60, "EM"),
    (2, 64, FM, 2, 3, 150, "M"), (2, 90, FM, 1, 2, 60, "EM"), (2, 92, FM, 1, 2, 20, "EM"), (2, 24, FM, 1, 3, 200, ""),
    (3, 4, EA, 3, 2, 400, "EM"), (3, 6, FM, 1, 2, 60, "EM"), (3, 8, EA, 2, 1, 200, "EM"), (3, 10, EA, 1, 3, 60, "EM"),
    (3, 12, EA, 2, 2, 60, "E"), (3, 14, FM, 1, 2, 40, "EM"), (3, 20, EA, 1, 2, 30, "EM"), (3, 22, EA, 1, 1, 10, "EM"),
    (3, 20, FM, 1, 1, 20, ""),
])
def test_sweeps_ahead_match_byte_kernel(ctx, dim, L, model, I, R, n, series):
    a = _run(ctx, gbmc.GBMC_KERNEL_AUTO, dim, L, model, I, R, n, series)
    b = _run(ctx, gbmc.GBMC_KERNEL_BYTES, dim, L, model, I, R, n, "EM")  # (takes no M without E)
    np.testing.assert_array_equal(a[0], b[0])
    for x, name in zip(a[1:], series):
        np.testing.assert_array_equal(x, b[1 + "EM".index(name)], err_msg=name)


@pytest.mark.parametrize("extra", [0, 1])
def test_as_many_copies_as_multiprocessors(ctx, extra):
    R = torch.cuda.get_device_properties(0).multi_processor_count + extra
    a, b = (_run(ctx, k, 2, 12, FM, 1, R, 30, "EM") for k in (gbmc.GBMC_KERNEL_AUTO, gbmc.GBMC_KERNEL_BYTES))
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)
