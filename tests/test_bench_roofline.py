"""The benchmark's roofline of a swept rate kernel is a share of what the card can issue, of executed instructions (no
GPU): at the measured 2.5 ms per 2^20 states of 53/325 below 1, and nothing where no capture of the kernel exists."""
import json
import os

import bench
from paper_2411_02640_gb300 import kx, synth


def test_swept_kernel_is_priced_by_what_it_executes(tmp_path, monkeypatch):
    path = synth.mechanism_file("gri_53_325", str(tmp_path))
    m = kx.Mechanism(path, cache_dir=str(tmp_path / "cache"), compile_only=1, lazy=1)
    for name in ("wdot_fp64", "wdot_mixed"):
        with open(os.path.join(bench.ROOT, "profiles", f"traffic_{name}_gri_53_325.json")) as f:
            rec = json.load(f)
        monkeypatch.setattr(m, "source_hash", lambda _: rec["source_hash"])
        r = bench.kernel_roofline(m, name, 1 << 20, 2.5, 2070.0)
        assert r["bound"] == "issue" and 0.3 < r["frac"] < 0.7
        monkeypatch.setattr(m, "source_hash", lambda _: "another build")
        r = bench.kernel_roofline(m, name, 1 << 20, 2.5, 2070.0)
        assert r["frac"] is None and r["method_work"]["rate"] > 0
    assert not bench.swept(m, "wdot_fp64_wc") and not bench.swept(m, "thermo")
    assert bench.kernel_roofline(m, "visc_fp64", 1 << 20, 1.3, 2070.0)["frac"] < 1
