"""The one-thread-per-state adjoint, whose sums over a species' reactions take the common factor 1/C_k once at the
end (above 16 species) or in each term, against the form with one log-space exponential per term."""
import numpy as np
import pytest

from paper_2411_02640_gb300 import synth
from tests.gpu_common import mechanism, to_device, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["h2o2_9_21", "gri_53_325", "large_160_900"])
@pytest.mark.parametrize("n", [1, 33, 129])
def test_against_one_exponential_per_term(name, n):
    torch = torch_cuda()
    m = synth.mechanism(name)
    rng = np.random.default_rng(n)
    T, p, Y = synth.make_states(m.n_species, synth.STATE_SPECS[name], 80 + n, n)
    Y[rng.random(Y.shape) < 0.2] = 0.0                    # absent species: C_k floored, R/C_k finite
    Y[0] += 0.1
    Y[2, n // 2] = -1e-7                                  # the sums carry the sign of C_k
    v = rng.standard_normal(Y.shape) * 10.0 ** rng.integers(-30, 30, n)
    d = to_device(torch, T, p, Y)
    v = torch.tensor(v, device="cuda")
    (gT, gY), (rT, rY) = (mechanism(name, vjp_layout=1, vjp_form=f).production_rates_vjp(*d, v) for f in (0, 1))
    # both to ~1e-10 of an entry's term scale; the entries of a state reach that of their largest
    assert float(((gY - rY).abs().amax(0) / rY.abs().amax(0)).max()) <= 1e-9
    assert torch.all(torch.isfinite(gT)) and torch.all((gT - rT).abs() <= 1e-9 * (rT.abs() + rY.abs().amax(0)))
