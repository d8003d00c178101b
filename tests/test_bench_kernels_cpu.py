"""Which kernel a benchmark line is about and the bytes its updates need, for the kernels that
keep copies on chip for many rounds or sweep a large lattice as tagged bit words."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_strips_of_bit_words():
    prof = {"stream_strips": (1, 1.0), "bitpack_convert": (2, 0.1)}
    for name in ("ising2d-L4096", "ising2d-L4096-bitpack"):
        w = dict(bench.WORKLOADS[name], L=1000 if name == "ising2d-L4096" else 448)
        assert bench.kernel_name(w, prof) == "stream_strips"
        # eight bytes for 32 sites of a word and its tag, read and written once per call
        assert bench.alg_bytes_per_update(w, "stream_strips") == 0.5 / 1000


def test_rounds_of_tempering():
    w = dict(bench.WORKLOADS["pt-ea3d-L8"])
    assert bench.kernel_name(w, {"pt_rounds": (2, 1.0)}) == "pt_rounds"
    assert bench.alg_bytes_per_update(w, "sweep_bits") == 2.0 / 10
    # 1024 x 32 copies of 512 sites, 10 sweeps: 102 rounds make 2^34 updates, the call has 100
    assert bench.alg_bytes_per_update(w, "pt_rounds") == 2.0 / (10 * 100)
    assert bench.alg_bytes_per_update(dict(w, rounds=400), "pt_rounds") == 2.0 / (10 * 102)
    # one sweep per round, a single instance: 2^13 sweeps
    assert bench.alg_bytes_per_update(dict(w, I=1, theta=1, rounds=10 ** 5), "pt_rounds") == 2.0 / 8192
