"""Mechanisms at the edges of the emitters' loops compile (no GPU)."""
import copy

import pytest

from paper_2411_02640_gb300 import kx, synth


def _compile(m, path, kernels):
    synth.write_mechanism(m, str(path))
    h = kx.Mechanism(str(path), cache_dir=str(path) + ".cache", compile_only=1, lazy=1)
    return {k: h.kernel_info(k) for k in kernels}


def test_adjoint_without_efficiency_lists(tmp_path):
    """Third-body reactions whose sum is [M] alone: no species has a third-body term."""
    m = copy.deepcopy(synth.mechanism("gri_53_325"))
    for r in m.reactions:
        r.efficiencies = {}
    assert any(r.uses_third_body() and r.collider is None for r in m.reactions)
    assert not any(r.uses_third_body() and r.collider is not None for r in m.reactions)
    _compile(m, tmp_path / "m.kxmech", ("vjp", "vjp_wc"))
