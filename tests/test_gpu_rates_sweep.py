"""The one-state-per-thread production rates with the straight-line float32 sweep (mechanisms up to 64 species
and 400 reactions): against the same kernel with every reaction in float pairs, at batch sizes around its blocks
of 256 and its warps, for every reaction form, absent species, undershoots and states outside the domain."""
import numpy as np
import pytest

from paper_2411_02640_gb300 import synth
from tests import toys
from tests.gpu_common import CACHE, mechanism, to_device, torch_cuda
from tests.test_gpu_reaction_kinds import _states, reactions

pytestmark = pytest.mark.gpu

# A negligible reaction runs below 2^-40 (9e-13) of its state's largest rate and float32 gives it to 1e-4: 325 of
# them are off by at most 3e-14 of that rate; the two kernels' float pairs, summed in different orders, by 1e-11
BAR = 1e-11


def _pair(name, tmp_path):
    if name != "kinds":
        return mechanism(name, rates_layout=1), mechanism(name, rates_layout=1, rates_negligible=1)
    from paper_2411_02640_gb300 import kx
    _, path = toys.toy("kinds", reactions(), str(tmp_path))
    return tuple(kx.Mechanism(path, cache_dir=CACHE, rates_layout=1, rates_negligible=g) for g in (0, 1))


def _draw(name, n, seed):
    if name == "kinds":
        return _states(n, seed)
    m = synth.mechanism(name)
    T, p, Y = synth.make_states(m.n_species, synth.STATE_SPECS[name], seed, n)
    T[:] = np.random.default_rng(seed).uniform(250.0, 3500.0, n)
    Y[:, ::5] = np.where((np.arange(m.n_species) % 3 == 0)[:, None], 0.0, Y[:, ::5])   # absent species
    return T, p, Y


@pytest.mark.parametrize("name", ["kinds", "h2o2_9_21", "gri_53_325"])
@pytest.mark.parametrize("n", [1, 31, 33, 255, 257, 1025])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_against_float_pairs(name, n, precision, tmp_path):
    torch = torch_cuda()
    a, b = _pair(name, tmp_path)
    T, p, Y = _draw(name, n, 40 + n)
    if n > 1:
        T[n // 2] = np.nan
    if n > 255:
        Y[1, 40] *= -0.01     # an undershoot: its warp takes the sweep with signs
    d = to_device(torch, T, p, Y, ld=n + 3)
    w, r = (m.production_rates(*d, precision=q)[:, :n].cpu().numpy() for m, q in ((a, precision), (b, "fp64")))
    ok = np.isfinite(T)
    assert np.all(np.isnan(w[:, ~ok])) and np.all(np.isfinite(w[:, ok]))
    W = np.asarray(a.W)[:, None]
    err = np.abs(W * (w - r))[:, ok].max(axis=0) / np.abs(W * r)[:, ok].max(axis=0)
    assert err.max() <= BAR, f"{err.max():.3e}"


@pytest.mark.parametrize("name", ["kinds", "gri_53_325"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_independent_of_neighbours(name, precision, tmp_path):
    """Without a large negative mass fraction in its warp (mixed: whatever its warp holds), a state's result is the
    same bits wherever it stands."""
    torch = torch_cuda()
    a, _ = _pair(name, tmp_path)
    T, p, Y = _draw(name, 700, 7)
    w = a.production_rates(*to_device(torch, T, p, Y), precision=precision)
    q = np.random.default_rng(1).permutation(700)[:413]
    v = a.production_rates(*to_device(torch, T[q], p[q], np.ascontiguousarray(Y[:, q])), precision=precision)
    assert torch.equal(v, w[:, torch.tensor(q, device="cuda")])
    Y[1, 100] = -Y[1, 100] - 1e-6
    v = a.production_rates(*to_device(torch, T, p, Y), precision=precision)
    lo, hi = (96, 128) if precision == "fp64" else (100, 101)
    assert torch.equal(v[:, :lo], w[:, :lo]) and torch.equal(v[:, hi:], w[:, hi:])
