"""Three-body reactions of a trace collider: [X] far below 1, where the rate without [X] is beyond float32's range of
the scale that the state's rates (with [X]) set."""
import numpy as np
import pytest

from paper_2411_02640_gb300 import kx
from paper_2411_02640_gb300.synth import P_ATM
from tests import toys
from tests.gpu_common import CACHE, to_device, torch_cuda, wdot_error

pytestmark = pytest.mark.gpu


def _padded(ns):
    specs = [("H", {"H": 1}, 2.5, 2.5e4, -0.5), ("O", {"O": 1}, 2.5, 3.0e4, 2.0), ("HO", {"H": 1, "O": 1}, 3.5, 4.0e3, 1.5),
             ("N2", {"N": 2}, 3.5, -1.0e3, 4.0)]
    return specs + [("X%d" % k, {"N": 2}, 3.5, -1.0e3, 4.0) for k in range(ns - 4)]


@pytest.mark.parametrize("ns,precision", [(4, "fp64"), (4, "mixed"), (70, "fp64")])
def test_trace_collider(ns, precision, tmp_path):
    torch = torch_cuda()
    import oracle
    rx = [toys.recomb("three_body", collider=3), toys.recomb("three_body", efficiencies={0: 2.0}, rate=(1e-30, 0.5, 1000.0))]
    _, path = toys.toy("trace%d" % ns, rx, str(tmp_path), specs=_padded(ns))
    n = 320
    rng = np.random.default_rng(8)
    T, p = rng.uniform(800.0, 2500.0, n), P_ATM * np.exp(rng.uniform(-3.0, 3.0, n))
    Y = rng.gamma(1.0, 1.0, (ns, n))
    Y /= Y.sum(axis=0)
    Y[3] = 10.0 ** -rng.uniform(0.0, 26.0, n)     # ([X] as a float pair: 48 bits down to 1e-28)
    Y[3, ::7] = 0.0
    ref = oracle.Oracle(path).production_rates(T, p, Y)
    mech = kx.Mechanism(path, cache_dir=CACHE, lazy=1, rates_layout=1)
    w = mech.production_rates(*to_device(torch, T, p, Y), precision=precision).cpu().numpy()
    assert np.all(np.isfinite(w))
    assert wdot_error(np.asarray(mech.W), w, ref).max() <= (2e-4 if precision == "mixed" else 1e-10)
