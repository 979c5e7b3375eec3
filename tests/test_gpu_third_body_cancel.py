"""Third-body sums that cancel: reactions with efficiencies of 0 in mixtures made of those species.  [X] =
e_default C_M + sum (e_k - e_default) C_k is then a small difference, of which the rate kernels' float32 estimates
hold only noise; their production rates against the same kernel with every reaction in float pairs."""
import copy

import numpy as np
import pytest

from paper_2411_02640_gb300 import kx, synth
from paper_2411_02640_gb300.synth import P_ATM
from tests import toys
from tests.gpu_common import CACHE, to_device, torch_cuda, wdot_error

pytestmark = pytest.mark.gpu


def _pair(name, tmp_path, bath):
    specs = [("H", {"H": 1}, 2.5, 2.5e4, -0.5), ("O", {"O": 1}, 2.5, 3.0e4, 2.0), ("HO", {"H": 1, "O": 1}, 3.5, 4.0e3, 1.5),
             ("N2", {"N": 2}, 3.5, -1.0e3, 4.0)] + [("X%d" % k, {"N": 2}, 3.5, -1.0e3, 4.0) for k in range(66)]
    kw = {"specs": specs} if name.endswith("70") else {}      # 70 species: table-driven loops, a vote of each warp
    if name in ("toy", "toy70"):
        # H + O + M <=> HO + M alone (its rate is the state's largest), and beside faster and slower reactions
        rx = [toys.recomb("three_body", efficiencies={k: 0.0 for k in bath})]
        _, path = toys.toy("bath1", rx, str(tmp_path), **kw)
    elif name in ("toys", "toys70"):
        rx = [toys.recomb("three_body", efficiencies={k: 0.0 for k in bath}), toys.recomb("elementary", rate=(1e-4, 0.5, 1000.0)),
              toys.recomb("falloff", rate=(1e9, 0.3, 400.0), rate_low=(1e12, 0.1, 100.0), efficiencies={k: 0.0 for k in bath})]
        _, path = toys.toy("bath3", rx, str(tmp_path), **kw)
    else:
        m = copy.deepcopy(synth.mechanism(name))
        for r in m.reactions:
            if r.uses_third_body() and r.collider is None:
                r.efficiencies = {**r.efficiencies, **{k: 0.0 for k in bath}}
        path = str(tmp_path / (name + "_bath.kxmech"))
        synth.write_mechanism(m, path)
    return tuple(kx.Mechanism(path, cache_dir=CACHE, lazy=1, rates_layout=1, rates_negligible=g) for g in (0, 1))


@pytest.mark.parametrize("bath", [(3,), (1, 3)])
@pytest.mark.parametrize("name", ["toy", "toys", "toy70", "toys70", "gri_53_325", "large_160_900"])
def test_bath_of_efficiency_zero(name, bath, tmp_path):
    torch_cuda()
    import torch
    a, b = _pair(name, tmp_path, bath)
    n, ns = 768, a.n_species
    rng = np.random.default_rng(5)
    T = rng.uniform(800.0, 2800.0, n)
    p = P_ATM * np.exp(rng.uniform(0.0, 3.0, n))
    rest = 10.0 ** -np.array([2.0, 6.0, 8.0, 10.0])[np.arange(n) // 192]      # a warp's states alike
    Y = rng.gamma(1.0, 1.0, (ns, n))
    Y[list(bath)] = 0.0
    Y *= rest / Y.sum(axis=0)
    f = rng.uniform(0.2, 0.8, n)
    for j, k in enumerate(bath):
        Y[k] = (1.0 - rest) * (1.0 if len(bath) == 1 else f if j == 0 else 1.0 - f)
    if name.endswith("70"):      # warps of one state each
        one = np.arange(n) // 32 * 32
        T, p, Y = T[one], p[one], np.ascontiguousarray(Y[:, one])
    d = to_device(torch, T, p, Y)
    r = b.production_rates(*d).cpu().numpy()
    for precision in ("fp64", "mixed") if ns <= 64 else ("fp64",):
        w = a.production_rates(*d, precision=precision).cpu().numpy()
        assert np.all(np.isfinite(w))
        # float32 for what is below 2^-40 of a state's largest rate; float pairs in another order: 1e-11
        assert wdot_error(np.asarray(a.W), w, r).max() <= 1e-11, rest[wdot_error(np.asarray(a.W), w, r) > 1e-11]
