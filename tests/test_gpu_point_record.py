"""Each production-rate and rates-of-progress kernel by itself records the smallest index of a point outside the
domain: at a batch above the crossover between the warp-cooperative and the thread-per-state kernels and at one below
it, for a bad T, a bad p and a zero sum of Y/W, with nothing else launched between the call and the check."""
import numpy as np
import pytest

from paper_2411_02640_gb300 import kx, synth
from tests.gpu_common import CACHE, MECHDIR, torch_cuda

pytestmark = pytest.mark.gpu


def _call(mech, which, T, p, Y):
    import torch
    if which == "noalloc":
        out = torch.empty_like(Y)
        mech.production_rates_noalloc(T, p, Y, out)
        return out
    if which.startswith("rop"):
        return mech.rates_of_progress(T, p, Y, precision=which[4:])
    return mech.production_rates(T, p, Y, precision=which)


@pytest.mark.parametrize("name", ["h2o2_9_21", "gri_53_325"])
@pytest.mark.parametrize("which", ["fp64", "mixed", "noalloc", "rop_fp64", "rop_mixed"])
@pytest.mark.parametrize("n", [301, 60001])
def test_recorded_and_nan(name, which, n):
    torch = torch_cuda()
    mech = kx.Mechanism(synth.mechanism_file(name, MECHDIR), cache_dir=CACHE, lazy=1)
    T, p, Y = synth.make_states_torch(mech.n_species, synth.STATE_SPECS[name], n, 9)
    _call(mech, which, T, p, Y)
    assert mech.last_point_status() == -1
    for at, (k, v) in zip((n - 1, 257, 97), (("T", np.nan), ("p", -1.0), ("Y", 0.0))):
        d = {"T": T.clone(), "p": p.clone(), "Y": Y.clone()}
        d[k][..., at] = v
        d["T"][n - 1] = np.inf      # a later one beside it
        out = _call(mech, which, d["T"], d["p"], d["Y"])
        assert mech.last_point_status() == at
        assert mech.last_point_status() == -1
        bad = torch.isnan(out).all(0).nonzero().flatten().tolist()
        assert bad == sorted({at, n - 1})
