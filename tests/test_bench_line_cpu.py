"""The line that the benchmark prints is short enough for a reader who keeps only the end of the
output, has every key of the result contract, and the whole record goes to a file on request."""
import json
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402


def _run_gpu(args, w, ws, rank, local, steps=None, warmup=None, e2e=True):
    steps = args.steps if steps is None else steps
    upd = float(bench.site_updates_per_step(w)) * steps
    kinds = ("sweep_bits", "pa_resample", "pa_record", "pa_reset", "init_spins", "observables", "bitpack_convert",
             "bitpack_strips", "swendsen_wang", "pt_exchange", "sweep_msc", "sweep_dcb_bits")
    r = dict(ms=278.48123456789 * steps, steps=steps, warmup=3, upd_all=upd, upd_local=upd, upd_prof=upd,
             ms_profiled=281.123456789 * steps, prof={k: (101 * steps, 270.123456789) for k in kinds}, launches=302 * steps,
             clocks={"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 40}, sm_count=152)
    if e2e:
        r["e2e"] = dict(seconds_per_step=0.31123456789, h2d=409600000, d2h=409616160, steps=steps,
                        step_seconds=[0.31123456789] * steps, clocks=r["clocks"])
    return r


@pytest.mark.parametrize("workload", ["pa-ising2d-L64", "pa-mixed-2d", "pt-ea3d-L8"])
def test_printed_line(workload, monkeypatch, capsys, tmp_path):
    learned = {"value": 20.09542550399999, "unit": "s", "config": {"Ls": [32, 64, 128, 256]}, "notes": "x" * 2000}
    monkeypatch.setattr(bench, "run_gpu", _run_gpu)
    monkeypatch.setattr(bench, "run_learned", lambda *a, **k: learned)
    monkeypatch.setattr(bench, "cpu_oracle_sample", lambda w: (0.0178120172578037, "a whole run, " * 20, 5.5))
    monkeypatch.setattr(bench, "cpu_oracle_all_cores", lambda w: (0.27566989405116277, 16, 5.7))
    path = tmp_path / "record.json"
    monkeypatch.setattr(sys, "argv", ["bench.py", "--steps", "20", "--warmup", "5", "--workload", workload,
                                      "--record", str(path)])
    bench.main()
    out = capsys.readouterr().out
    assert out.count("\n") == 1 and len(out) < 2500  # some 3000 characters of output are kept
    d = json.loads(out)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "cpu_baseline"):
        assert k in d, k
    for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert k in d["e2e"]
    for k in ("bound", "achieved", "peak", "unit", "frac", "traffic"):
        assert k in d["roofline"]
    assert d["clocks"]["reasons"] == ["sw_power_cap"]
    full = json.loads(path.read_text())
    assert full["value"] == d["value"] > 0 and "kernels" in full and full["e2e"]["step_ms"]
    if workload == "pa-ising2d-L64":
        assert set(d["secondary"]) == set(bench.SECONDARY) | {"pa-learned"}
        assert full["secondary"]["pa-learned"] == learned
