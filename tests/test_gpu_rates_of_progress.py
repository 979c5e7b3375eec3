"""Rates of progress on both sides of the batch size from which one thread per
state is faster: small batches run the warp-cooperative kernel, for either
precision, large ones one thread per state."""
import numpy as np
import pytest

from paper_2411_02640_gb300 import synth
from tests.gpu_common import mechanism, oracle, to_device, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("name,n", [("h2o2_9_21", 1), ("h2o2_9_21", 1001), ("gri_53_325", 33), ("gri_53_325", 1289),
                                    ("large_160_900", 131)])
def test_small_batches_against_oracle(name, n, precision):
    torch = torch_cuda()
    m = synth.mechanism(name)
    T, p, Y = synth.make_states(m.n_species, synth.STATE_SPECS[name], 900, n)
    if n > 100:
        Y[:, 7] = np.where(np.arange(m.n_species) % 3 == 0, 0.0, Y[:, 7])   # absent species
        Y[1, 9] *= -0.1                                                      # an undershoot
        T[11] = -1.0                                                         # outside the domain
    mech = mechanism(name)
    q = mech.rates_of_progress(*to_device(torch, T, p, Y, ld=n + 5), precision=precision)[:, :n].cpu().numpy()
    ok = T > 0
    o = oracle(name)
    T2, p2, Y2 = T[ok], p[ok], np.ascontiguousarray(Y[:, ok])
    gross = o.reaction_gross(T2, p2, Y2)
    rel = np.abs(q[:, ok] - o.rates_of_progress(T2, p2, Y2)) / np.where(gross > 0, gross, 1.0)
    assert rel.max() <= 1e-10, f"{rel.max():.3e}"      # both precisions: the float-pair kernel
    assert np.all(np.isnan(q[:, ~ok]))
    assert mech.last_point_status() == (11 if n > 100 else -1)


@pytest.mark.parametrize("name,low,high", [("h2o2_9_21", 2000, 20000), ("gri_53_325", 9000, 60000)])
def test_choice_by_batch_size(name, low, high):
    """A large batch runs the thread-per-state kernel bit for bit; a small one agrees with it within the
    two kernels' bound (1e-10 of the reaction's gross scale)."""
    torch = torch_cuda()
    m = synth.mechanism(name)
    auto, tps = mechanism(name), mechanism(name, rates_layout=1)
    for n in (low, high):
        T, p, Y = synth.make_states(m.n_species, synth.STATE_SPECS[name], 1700, n)
        d = to_device(torch, T, p, Y)
        a, b = auto.rates_of_progress(*d), tps.rates_of_progress(*d)
        if n == high:
            assert torch.equal(a, b)
        else:
            i = slice(0, 200)
            gross = torch.tensor(oracle(name).reaction_gross(T[i], p[i], np.ascontiguousarray(Y[:, i])), device="cuda")
            assert float(((a - b)[:, i].abs() / gross).max()) <= 1e-10
