"""Production rates of states with negative mass fractions (transport undershoots) through the float32 sweep, which
gives them the signs of the concentration products: against the same kernel with every reaction in float pairs."""
import numpy as np
import pytest

from paper_2411_02640_gb300 import kx, synth
from tests import toys
from tests.gpu_common import CACHE, mechanism, to_device, torch_cuda
from tests.test_gpu_reaction_kinds import _states, reactions

pytestmark = pytest.mark.gpu


def _handles(name, tmp_path):
    if name == "kinds":
        rx = reactions() + [toys.recomb("three_body", efficiencies={1: 0.0, 3: 0.0}, rate=(1e8, 0.2, 500.0)),
                            toys.recomb("falloff", collider=0, rate=(1e9, 0.3, 400.0), rate_low=(1e12, 0.1, 100.0)),
                            toys.recomb("three_body", collider=2, rate=(3e9, -0.5, 200.0))]
        _, path = toys.toy("kinds_signs", rx, str(tmp_path))
        return tuple(kx.Mechanism(path, cache_dir=CACHE, lazy=1, rates_layout=1, rates_negligible=g) for g in (0, 1))
    return mechanism(name, rates_layout=1), mechanism(name, rates_layout=1, rates_negligible=1)


def _draw(name, n, seed):
    rng = np.random.default_rng(seed)
    if name == "kinds":
        T, p, Y = _states(n, seed)
    else:
        m = synth.mechanism(name)
        T, p, Y = synth.make_states(m.n_species, synth.STATE_SPECS[name], seed, n)
        T[:] = rng.uniform(400.0, 3000.0, n)
    return rng, T, p, Y


def _err(W, w, r):
    W = np.asarray(W)[:, None]
    return np.abs(W * (w - r)).max(axis=0) / np.abs(W * r).max(axis=0)


@pytest.mark.parametrize("name", ["kinds", "h2o2_9_21", "gri_53_325"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("size", [1e-12, 1e-6, 1e-3, 0.3])
def test_one_percent_negative(name, precision, size, tmp_path):
    torch = torch_cuda()
    a, b = _handles(name, tmp_path)
    rng, T, p, Y = _draw(name, 2049, 11)
    share = 0.1 if name == "kinds" else 0.01
    Y = np.where(rng.random(Y.shape) < share, -size * rng.random(Y.shape), Y)
    ok = (Y / np.asarray(a.W)[:, None]).sum(axis=0) > 1e-4      # sum Y/W > 0: inside the domain, and not cancelled
    T, p, Y = T[ok], p[ok], np.ascontiguousarray(Y[:, ok])
    assert (Y < 0).any(axis=0).sum() > 100
    d = to_device(torch, T, p, Y)
    w, r = a.production_rates(*d, precision=precision).cpu().numpy(), b.production_rates(*d).cpu().numpy()
    assert np.all(np.isfinite(w))
    # as without negative mass fractions: float32 below 2^-40 of the largest rate, float pairs in another order
    assert _err(a.W, w, r).max() <= 1e-11


@pytest.mark.parametrize("name", ["kinds", "gri_53_325"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_beside_undershoots(name, precision, tmp_path):
    """States keep their bits beside states with undershoots, and those theirs wherever they stand."""
    torch = torch_cuda()
    a, _ = _handles(name, tmp_path)
    rng, T, p, Y = _draw(name, 700, 12)
    w = a.production_rates(*to_device(torch, T, p, Y), precision=precision)
    hit = np.arange(0, 700, 7)
    Y[1, hit] = -1e-7
    v = a.production_rates(*to_device(torch, T, p, Y), precision=precision)
    rest = torch.tensor(np.setdiff1d(np.arange(700), hit), device="cuda")
    assert torch.equal(v[:, rest], w[:, rest])
    alone = a.production_rates(*to_device(torch, T[hit], p[hit], np.ascontiguousarray(Y[:, hit])), precision=precision)
    assert torch.equal(alone, v[:, torch.tensor(hit, device="cuda")])
