"""Rates of progress whose float64 value overflows: infinities of the right sign from the warp-cooperative kernel of
small batches as from the thread-per-state one (cold states of the synthetic mechanisms reach 1e308)."""
import numpy as np
import pytest

from paper_2411_02640_gb300 import synth
from tests.gpu_common import mechanism, oracle, to_device, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["h2o2_9_21", "gri_53_325", "large_160_900"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_overflow_is_infinite(name, precision):
    torch = torch_cuda()
    n = 97
    T, p, Y = synth.make_states(synth.mechanism(name).n_species, synth.STATE_SPECS[name], 21, n)
    T[:] = np.linspace(100.0, 220.0, n)
    d = to_device(torch, T, p, Y)
    q, r = (mechanism(name, **o).rates_of_progress(*d, precision=precision).cpu().numpy() for o in ({}, {"rates_layout": 1}))
    over = np.isinf(r)
    assert over.sum() > 50 and np.array_equal(q[over], r[over])
    assert np.all(np.isfinite(r[~over]) & (np.isfinite(q[~over]) | (np.abs(r[~over]) > 1e300)))
    ref = oracle(name).rates_of_progress(T, p, Y)      # (its products may overflow on the way to a finite rate)
    with np.errstate(invalid="ignore"):
        assert np.all(np.isinf(ref[over]) | np.isnan(ref[over]) | (np.abs(ref[over]) > 1e307))
