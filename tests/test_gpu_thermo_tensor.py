"""The tensor-core thermo kernel: ragged tiles, both sides of T_mid and
temperatures far outside the blocks' range (the polynomials are evaluated as
given there too), unnormalised, negative and non-finite mass fractions, and
mechanisms whose species have different T_mid."""
import dataclasses

import numpy as np
import pytest

from paper_2411_02640_gb300 import kx, synth
from tests.gpu_common import CACHE, mechanism, oracle, to_device, torch_cuda

pytestmark = pytest.mark.gpu


def check(mech, ora, m, T, p, Y):
    torch = torch_cuda()
    cp, h = (t.cpu().numpy() for t in mech.thermo(*to_device(torch, T, p, Y, ld=T.shape[0] + 3)))
    cp_r, h_r = ora.thermo(T, p, Y)
    for i in range(T.shape[0]):
        t = ora.species_thermo(T[i])
        w = np.abs(Y[:, i]) * synth.R_U / m.W
        assert abs(cp[i] - cp_r[i]) <= 1e-12 * np.sum(w * np.abs(t["cp_R"])), i
        assert abs(h[i] - h_r[i]) <= 1e-12 * np.sum(w * np.abs(t["h_RT"])) * T[i], i


@pytest.mark.parametrize("name,n", [("h2o2_9_21", 1), ("h2o2_9_21", 129), ("gri_53_325", 257), ("large_160_900", 140)])
def test_against_oracle(name, n):
    m = synth.mechanism(name)
    T, p, Y = synth.make_states(m.n_species, synth.STATE_SPECS[name], 60, n)
    if n > 100:
        T[:8] = (100.0, 199.0, 999.9999, 1000.0, 1000.0001, 4000.0, 4500.0, 6000.0)
        Y[:, 20:30] *= 1e-7
        Y[:, 30:40] *= 1e7
        Y[3, 40:50] *= -0.05
        Y[1:4, 50:60] = 0.0
    check(mechanism(name), oracle(name), m, T, p, Y)


@pytest.mark.parametrize("mids", [2, 4, 6])
def test_different_mid_temperatures(tmp_path, mids):
    """Two and four distinct T_mid (rows of each group chosen per state); six fall back to one thread per state."""
    import oracle as ora
    m = synth.mechanism("h2o2_9_21")
    nasa_T = m.nasa_T.copy()
    nasa_T[:, 1] = 1000.0 + 100.0 * (np.arange(m.n_species) % mids)
    m = dataclasses.replace(m, name=f"mids{mids}", nasa_T=nasa_T)
    path = str(tmp_path / "m.kxmech")
    synth.write_mechanism(m, path)
    T, p, Y = synth.make_states(m.n_species, synth.STATE_SPECS["h2o2_9_21"], 0, 200)
    T[:6] = (1000.0, 1100.0, 1150.0, 1199.9, 1300.0, 1500.0)
    check(kx.Mechanism(path, cache_dir=CACHE), ora.Oracle(path, nthreads=4), m, T, p, Y)


def test_points_outside_the_domain():
    torch = torch_cuda()
    T, p, Y = synth.make_states(53, synth.STATE_SPECS["gri_53_325"], 5, 150)
    T[4], p[6], Y[2, 8], Y[:, 9] = np.nan, -1.0, np.nan, 0.0
    mech = mechanism("gri_53_325")
    cp, h = (t.cpu().numpy() for t in mech.thermo(*to_device(torch, T, p, Y)))
    assert mech.last_point_status() == 4
    assert np.all(np.isnan(cp[[4, 6, 8]])) and np.all(np.isnan(h[[4, 6, 8]]))
    assert cp[9] == 0.0 and h[9] == 0.0
    rest = np.setdiff1d(np.arange(150), [4, 6, 8])
    assert np.all(np.isfinite(cp[rest])) and np.all(np.isfinite(h[rest]))
