"""The tensor-core kernels' bounded waits (host-side text checks): a wait that runs out makes its results nan and
records the point in every block and warp that it concerns, and none stores what it did not wait for."""
import re

import pytest

from paper_2411_02640_gb300 import kx, synth


@pytest.mark.parametrize("kernel", ["visc_fp64", "visc_mixed", "diff_fp64", "diff_mixed", "thermo"])
def test_failed_wait_is_reported(kernel, tmp_path):
    path = synth.mechanism_file("gri_53_325", str(tmp_path))
    src = kx.Mechanism(path, cache_dir=str(tmp_path / "cache"), compile_only=1, lazy=1).kernel_source(kernel)
    lines = [line.strip() for line in src.split("\n") if len(line) < 400]
    # every guard of a store of results looks at the waits
    guards = [line for line in lines if re.search(r"in && !bad && !gen", line)]
    assert guards and all("&& ok" in line for line in guards)
    # ... its own and, where it reads the other groups' shared values, theirs
    i = lines.index("if (!ok) failed = 1;")
    assert lines[i + 1] == "KX_COMPUTE_SYNC;" and "ok && !failed" in lines[i + 2]
    # reported by every block (gridDim.y of them may share a tile's rows), not only the first of a column
    i = lines.index("if (!ok && in) {")
    report = " ".join(lines[i:i + 8])
    assert "atomicMin(&kx_bad_first" in report and "KX_NAN" in report
    assert not any("cy == 0" in line and "!ok" in line for line in lines)
