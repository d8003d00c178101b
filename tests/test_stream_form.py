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
