"""Mechanisms at the edges of the emitters' loops compile (no GPU needed) and run."""
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


@pytest.mark.parametrize("name", ["h2o2_9_21", "gri_53_325", "large_160_900"])
def test_without_reactions(name, tmp_path):
    """An inert mixture: the rate kernels write zeros, thermo and transport work."""
    m = copy.deepcopy(synth.mechanism(name))
    m.reactions = []
    _compile(m, tmp_path / "m.kxmech", kx.KERNELS)


def test_one_species(tmp_path):
    from tests import toys
    _, path = toys.toy("one", [], str(tmp_path), specs=[("N2", {"N": 2}, 3.5, -1.0e3, 4.0)])
    h = kx.Mechanism(path, cache_dir=str(tmp_path / "cache"), compile_only=1, lazy=1)
    assert all(h.kernel_info(k)["registers"] > 0 for k in kx.KERNELS)


@pytest.mark.gpu
def test_inert_mixture_runs(tmp_path):
    """Rates zero (in both rate kernels' ranges), thermo and transport as with the reactions."""
    from tests.gpu_common import CACHE, torch_cuda
    torch = torch_cuda()
    m = copy.deepcopy(synth.mechanism("h2o2_9_21"))
    synth.write_mechanism(m, str(tmp_path / "full.kxmech"))
    m.reactions = []
    synth.write_mechanism(m, str(tmp_path / "inert.kxmech"))
    h, full = (kx.Mechanism(str(tmp_path / f), cache_dir=CACHE) for f in ("inert.kxmech", "full.kxmech"))
    for n in (33, 20001):
        T, p, Y = synth.make_states_torch(9, synth.STATE_SPECS["h2o2_9_21"], n, 4)
        for precision in ("fp64", "mixed"):
            assert torch.count_nonzero(h.production_rates(T, p, Y, precision=precision)) == 0
        for a, b in zip(h.thermo(T, p, Y) + h.transport(T, p, Y), full.thermo(T, p, Y) + full.transport(T, p, Y)):
            assert torch.equal(a, b)


@pytest.mark.parametrize("name,most", [("h2o2_9_21", 32), ("gri_53_325", 64), ("53_400", 64)])
def test_noalloc_kernel_keeps_its_vectors_in_the_scratch(name, most, tmp_path):
    """Almost no local memory per thread, which the driver would back for every resident thread of the device:
    32 bytes at 53/325, 24 at 53 species and 400 reactions."""
    m = copy.deepcopy(synth.mechanism("gri_53_325" if name == "53_400" else name))
    if name == "53_400":
        m.reactions = m.reactions + m.reactions[:75]
    k = _compile(m, tmp_path / "m.kxmech", ("wdot_fp64_noalloc",))
    assert k["wdot_fp64_noalloc"]["local_bytes"] <= most
