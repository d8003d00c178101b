"""How the bit-stream kernel spreads a launch over the device, worked out on the host: every job
of a launch counts, copies too large for a one-warp team included, and the forms that the GPU
tests of the kernel mean to run are the ones it takes on 152 multiprocessors."""
import pytest

from paper_1709_04394_gb300 import build as gbuild
from paper_1709_04394_gb300 import gbmc


@pytest.fixture(scope="module", autouse=True)
def _library():
    gbuild.build()


def form(*lattices, **kw):
    return gbmc.gbmc_test_stream_form(lattices, **kw)


@pytest.mark.parametrize("big,small", [((2, 160, 1), (2, 24, 1, 2000)), ((2, 180, 1), (2, 40, 1, 5000)),
                                       ((3, 30, 4), (3, 8, 4, 500)), ((3, 32, 1), (3, 10, 1, 9000))])
def test_a_large_copys_job_counts_among_others(big, small):
    few, many = form((*big, 200), small), form((*big, 20000), small)
    # a hundred times the work of the job that makes up most of the launch
    assert many.cycles > 20 * few.cycles
    # no form is taken whose estimate leaves the job out: together they cost what the large one alone does
    assert few.cycles > 0.6 * form((*big, 200)).cycles


@pytest.mark.parametrize("copies,expected", [
    ((2, 40, 1, 201), (1, 4, 128)), ((2, 24, 1, 1513), (1, 2, 32)), ((2, 24, 1, 9001), (1, 1, 32)),
    ((2, 96, 1, 2161), (2, 1, 160)), ((2, 12, 1, 70001), (4, 1, 32)), ((3, 10, 3, 6603), (4, 1, 32)),
    ((3, 4, 7, 44491), (2, 1, 32)), ((3, 14, 1, 201), (1, 2, 96)), ((2, 204, 1, 481), (1, 1, 672)),
])
def test_one_lattice_from_few_copies_to_many(copies, expected):
    f = form(copies)
    assert (f.copies_per_thread, f.threads_per_word, f.team[0]) == expected


def test_sizes_annealed_together_share_the_device():
    # teams of one warp for all, two copies per thread, largest lattice first
    f = form((2, 24, 1, 20000), (2, 40, 1, 10000), (2, 96, 1, 4000))
    assert (f.copies_per_thread, f.threads_per_word, list(f.team[:3]), list(f.groups[:3])) == (2, 1, [32] * 3, [1, 1, 3])
