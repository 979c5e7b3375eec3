"""The tensor-core transport kernels where they can go wrong: ragged tiles of
128 states, temperatures at and beyond the ends of their basis (200 and 4000 K,
beyond which states are evaluated pair by pair), nearly pure states (whose own
row is evaluated pair by pair), unnormalised and negative mass fractions,
states outside the domain, and mechanisms of one to ten rows of 16."""
import numpy as np
import pytest

from paper_2411_02640_gb300 import synth
from tests.gpu_common import mechanism, oracle, to_device, torch_cuda

pytestmark = pytest.mark.gpu

NAMES = ("h2o2_9_21", "gri_53_325", "large_160_900")


def states(name, n, start=400):
    return synth.make_states(synth.mechanism(name).n_species, synth.STATE_SPECS[name], start, n)


def check(name, T, p, Y, precision, ld_pad=0):
    torch = torch_cuda()
    n = T.shape[0]
    mech = mechanism(name)
    Td, pd, Yd = to_device(torch, T, p, Y, ld=n + ld_pad)
    mu, lam, D = (t.cpu().numpy() for t in mech.transport(Td, pd, Yd, precision=precision))
    mu_r, lam_r, D_r = oracle(name).transport(T, p, Y)
    tol = 1e-12 if precision == "fp64" else 5e-6
    np.testing.assert_allclose(mu, mu_r, rtol=tol)
    np.testing.assert_allclose(lam, lam_r, rtol=tol)
    # the oracle forms (Wbar - X_k W_k)/Wbar literally: float64's rounding over the partners' share
    f = Y / Y.sum(axis=0)
    share = np.maximum(np.abs(1.0 - f), 1e-300)
    assert np.all(np.abs(D[:, :n] / D_r - 1) <= tol + 2e-15 / share)
    assert mech.last_point_status() == -1


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("name,n", [("h2o2_9_21", 1), ("h2o2_9_21", 129), ("gri_53_325", 127), ("gri_53_325", 128),
                                    ("gri_53_325", 40001), ("large_160_900", 130)])
def test_ragged_tiles(name, n, precision):
    """Also more tiles than blocks (40001 states: 313 tiles), and the row-sharing of few tiles."""
    T, p, Y = states(name, n)
    if n > 4000:
        # the oracle on a sample of the tiles' ends and middles
        torch = torch_cuda()
        mech = mechanism(name)
        Td, pd, Yd = to_device(torch, T, p, Y)
        out = [t.cpu().numpy() for t in mech.transport(Td, pd, Yd, precision=precision)]
        i = np.unique(np.concatenate([np.arange(0, n, 257), [127, 128, n - 1]]))
        ref = oracle(name).transport(T[i], p[i], np.ascontiguousarray(Y[:, i]))
        for a, b in zip(out, ref):
            np.testing.assert_allclose(a[..., i], b, rtol=1e-12 if precision == "fp64" else 5e-6)
    else:
        check(name, T, p, Y, precision, ld_pad=7)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("name", NAMES)
def test_temperature_range_and_nearly_pure(name, precision):
    T, p, Y = states(name, 300)
    ends = np.array([150.0, 199.999, 200.0, 200.001, 999.9, 1000.0, 3999.99, 4000.0, 4000.01, 5000.0])
    T[:10], T[130:140] = ends, ends
    for q, eps in enumerate((0.3, 1e-1, 3e-2, 1e-3, 1e-6)):
        for k in range(4):   # species k fills 1 - eps of the state
            i = 20 + 4 * q + k
            Y[:, i] *= eps / (Y[:, i].sum() - Y[k, i])
            Y[k, i] = 1.0 - eps
    Y[:, 60:70] *= 1e-6
    Y[:, 70:80] *= 1e6
    Y[2:5, 80:90] = 0.0
    check(name, T, p, Y, precision)


def test_outside_the_domain():
    """Non-finite and vanishing mass fractions, and bad T or p: NaN for those points alone; a pure
    species gets its self-diffusion coefficient."""
    torch = torch_cuda()
    name = "gri_53_325"
    T, p, Y = states(name, 200)
    T[3], p[5], T[7], Y[4, 9], Y[4, 11] = -1.0, 0.0, np.nan, np.inf, np.nan
    Y[:, 13] = 0.0
    Y[:, 15] = 0.0
    Y[6, 15] = 1.0
    bad = [3, 5, 7, 9, 11, 13]
    ok = np.setdiff1d(np.arange(200), bad)
    mech = mechanism(name)
    for precision in ("fp64", "mixed"):
        out = [t.cpu().numpy() for t in mech.transport(*to_device(torch, T, p, Y), precision=precision)]
        assert mech.last_point_status() == 3
        ref = oracle(name).transport(T[ok], p[ok], np.ascontiguousarray(Y[:, ok]))
        for a, b in zip(out, ref):
            assert np.all(np.isnan(a[..., bad])) and np.all(np.isfinite(a[..., ok]))
            np.testing.assert_allclose(a[..., ok], b, rtol=1e-12 if precision == "fp64" else 5e-6)


@pytest.mark.parametrize("name", ["h2o2_9_21", "gri_53_325"])
def test_negative_mass_fractions(name):
    """Undershoots of a transport step: against the pair-by-pair kernel, relative to the sums of absolute terms
    (at most (1 + 2 e)/(1 - 2 e) of the signed ones for a share e = 0.02 of negative values)."""
    torch = torch_cuda()
    T, p, Y = states(name, 260)
    rng = np.random.default_rng(3)
    neg = rng.random(Y.shape) < 0.1
    Y = np.where(neg, -Y * 0.02, Y)
    d = to_device(torch, T, p, Y)
    a = [t.cpu().numpy() for t in mechanism(name).transport(*d)]
    b = [t.cpu().numpy() for t in mechanism(name, tr_layout=3).transport(*d)]
    for x, y in zip(a, b):
        np.testing.assert_allclose(x, y, rtol=2e-12)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_same_bits_alone_and_in_a_batch(precision):
    """A state's results do not depend on its tile, on the blocks that share a tile's rows or on the leading dimension."""
    torch = torch_cuda()
    name, n = "gri_53_325", 30000
    T, p, Y = to_device(torch, *states(name, n))
    mech = mechanism(name)
    whole = mech.transport(T, p, Y, precision=precision)
    for a, b in ((0, 1), (100, 228), (777, 2777), (29000, 30000)):
        part = mech.transport(T[a:b].contiguous(), p[a:b].contiguous(), Y[:, a:b].contiguous(), precision=precision)
        for x, y in zip(part, whole):
            assert torch.equal(x, y[..., a:b])


@pytest.mark.parametrize("kernel", ["visc_fp64", "diff_fp64", "thermo"])
@pytest.mark.parametrize("name", ["gri_53_325", "large_160_900"])
def test_like_mass_fractions(name, kernel):
    """All of a kernel's scaled mass fractions near their largest: the largest sums that its products' exact integer
    accumulation has to hold (108 of the 64 that float32 holds, for a row of 160/900's viscosity)."""
    import re
    torch = torch_cuda()
    mech = mechanism(name)
    src = mech.kernel_source(kernel)
    ecol = np.array([int(v) for v in re.search(r"kx_ecol\[\d+\] = \{(.*?)\}", src).group(1).split(",") if v.strip()])
    T, p, Y = states(name, 256)
    rng = np.random.default_rng(2)
    u = 1.0 - rng.uniform(0.0, 0.02, Y.shape) * (np.arange(256) % 2)        # every other state: all alike
    Y = u * 2.0 ** -(ecol[:Y.shape[0], None] + 8.0)                        # the products' v: u (unnormalised states)
    d = to_device(torch, T, p, Y)
    if kernel == "thermo":
        got, ref = mech.thermo(*d), oracle(name).thermo(T, p, Y)
        ref = (ref[0], ref[1])
    else:
        got, ref = mech.transport(*d), oracle(name).transport(T, p, Y)
        got, ref = (got[:2], ref[:2]) if kernel == "visc_fp64" else (got[2:], ref[2:])
    for a, b in zip(got, ref):
        a = a.cpu().numpy()
        err = np.abs(a - b) / (np.abs(b) if kernel != "thermo" else np.abs(b).max())
        assert err.max() <= 1e-13, f"{err.max():.2e}"


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("name", NAMES)
@pytest.mark.parametrize("share", [1.0, 0.45, 0.1])
def test_outside_the_basis(name, precision, share):
    """Tiles of states below 200 K or above 4000 K, all of them or among others: a warp per state, its lanes over the
    rows; nearly pure and pure states."""
    T, p, Y = states(name, 275)
    out = np.where(np.arange(275) % 2, 4000.0 + 10.0 * np.arange(275), 199.0 - 0.3 * np.arange(275))
    T = np.where(np.random.default_rng(7).random(275) < share, out, T)
    T[3] = 4500.0
    for q, eps in enumerate((0.45, 1e-3, 1e-9)):
        for k in range(4):   # species 2 k fills 1 - eps of the state
            i = 20 + 4 * q + k
            Y[:, i] *= eps / (Y[:, i].sum() - Y[2 * k, i])
            Y[2 * k, i] = 1.0 - eps
    Y[-3:, 80:90] = 0.0
    check(name, T, p, Y, precision, ld_pad=5)
    Y[:, 3] = 0.0
    Y[4, 3] = 1.0
    torch = torch_cuda()
    out = [t.cpu().numpy() for t in mechanism(name).transport(*to_device(torch, T, p, Y), precision=precision)]
    ref = oracle(name).transport(T[3:4], p[3:4], np.ascontiguousarray(Y[:, 3:4]))
    for a, b in zip(out, ref):
        np.testing.assert_allclose(a[..., 3:4], b, rtol=1e-12 if precision == "fp64" else 5e-6)
