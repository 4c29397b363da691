"""The psi_fp64 option: psi of FP32 storage to double precision.  The float it gives is within
half a unit in the last place of psi, up to the rounding errors of FP64 arithmetic: about ten
operations (2^-53 each, taken as 2^-49 together) on Eq. 30's bracket R T Z - a rho - 1/3, whose
terms may cancel (ratio of their sum to the bracket)."""
import numpy as np
import pytest

import oracle
from tests import pairs

gpu = pytest.mark.gpu


def wide_psi(rho, c):
    """psi and the cancellation ratio in numpy's long double (64 bits or more)."""
    L = np.longdouble
    r = rho.astype(L)
    x = L(pairs.B / 4.0) * r
    with np.errstate(all="ignore"):
        z = (1 + x * (1 + x * (1 - x))) / (1 - x) ** 3
        brk = L(c["T"]) * z - L(c["a"]) * r - L(1) / L(3)
        ratio = (abs(L(c["T"]) * z) + L(c["a"]) * r + L(1) / L(3)) / abs(brk)
        arg = L(2.0) / L(c["G"]) * r * brk
        return np.where(arg > 0, np.sqrt(arg), L(0)), ratio


def vanishing_density(c):
    """The density in (0.3, 0.9) above which psi is 0, by bisection."""
    lo, hi = 0.3, 0.9
    assert wide_psi(np.array([lo]), c)[0] > 0 and wide_psi(np.array([hi]), c)[0] == 0
    while hi - lo > 1e-13:
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if wide_psi(np.array([mid]), c)[0][0] > 0 else (lo, mid)
    return lo


def densities(c):
    """Floats over the whole range of use, up to and beyond x = 3/4, dense next to psi = 0."""
    rng = np.random.default_rng(5)
    zero = vanishing_density(c)
    rho = np.concatenate([np.exp(rng.uniform(np.log(1e-4), np.log(0.9), 400000)),
                          np.geomspace(1e-38, 1e-4, 20000),
                          rng.uniform(zero - 1e-3, zero, 200000)])
    return np.unique(rho.astype(np.float32)).astype(np.float64)


def excess(got, rho, c):
    """How far `got` is from psi, over half a unit in the last place and FP64's errors."""
    ref, ratio = wide_psi(rho, c)
    half = np.spacing(np.maximum(ref.astype(np.float32), np.float32(1e-30))).astype(float) / 2
    ok = (ratio < 2.0 ** 40) & (ref > 0)
    return (np.abs(got - ref)[ok] / (half + ref * ratio * 2.0 ** -49)[ok]).astype(float)


@gpu
@pytest.mark.parametrize("tr", [0.5, 0.6, 0.7, 0.8, 0.9])
def test_option_gives_the_nearest_float(tr):
    c = pairs.case(8, 8, tr=tr)
    rho = densities(c)
    with pairs.gpu_lattice(c, "fp32", psi_fp64=True) as L:
        e = excess(L.eval_psi(rho), rho, c)
    assert len(e) > 300000 and e.max() <= 1.0, (e.max(), int((e > 1).sum()))
    with pairs.gpu_lattice(c, "fp32") as L:  # plain FP32 does not
        assert excess(L.eval_psi(rho), rho, c).max() > 10.0


@gpu
def test_where_fp64_decides():
    """Zero, subnormals, x = 1 and beyond, infinities, NaN: FP64 arithmetic, rounded."""
    from tests.test_gpu_fp64_edges import ieee_psi
    for G in (-1.0, 1.0):
        c = pairs.case(8, 8, tr=0.7, G=G)
        rho = np.array([0.0, -0.1, 1e-44, 1e-39, 0.75, 0.7500001, 0.999, 1.0, 1.25, 7.0, -3.0,
                        3e38, np.inf, -np.inf, np.nan])
        rho = rho.astype(np.float32).astype(np.float64)
        with pairs.gpu_lattice(c, "fp32", psi_fp64=True) as L:
            got = L.eval_psi(rho)
        with np.errstate(all="ignore"):
            ref = ieee_psi(rho, c).astype(np.float32).astype(np.float64)
        assert np.array_equal(got, ref), (got, ref)


def vanishing(c, shape, seed):
    """Columns of densities at psi = 0 (floats within 1e-6 below it) between columns of 0.1."""
    rho = vanishing_density(c) - np.random.default_rng(seed).uniform(0.0, 1e-6, shape)
    rho = np.where(np.arange(shape[1])[None, :] % 3 == 0, 0.1, rho)
    return rho.astype(np.float32).astype(np.float64)


def test_plain_fp32_psi_misses_where_psi_vanishes():
    """The premise of the next test, on the densities it uses: FP32 arithmetic on the bracket
    leaves psi wrong by more than 1e-4 there (no GPU)."""
    c = pairs.case(96, 20, tr=0.8)
    rho = vanishing(c, (20, 96), 3)
    f = np.float32
    x = f(1.0) * rho.astype(f)
    z = (f(1) + x * (f(1) + x * (f(1) - x))) / ((f(1) - x) * (f(1) - x) * (f(1) - x))
    arg = f(-2) * rho.astype(f) * (f(c["T"]) * z - f(c["a"]) * rho.astype(f) - f(1 / 3))
    got = np.sqrt(np.maximum(arg, f(0)))
    assert np.max(np.abs(got - wide_psi(rho, c)[0])) > 1e-4


@gpu
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("nx,vec,rows,persistent", [
    (96, 2, 1, 0), (96, 2, 2, 0), (96, 2, 7, 0), (300, 2, 1, 0), (300, 2, 5, 0), (96, 1, 4, 0),
    (300, 1, 4, 0), (96, 2, 7, 2), (300, 2, 5, 2)])
def test_step_uses_it(monkeypatch, nx, vec, rows, persistent, walls):
    """One step of a lattice whose nodes hold rest populations only, so that FP32 sums them to
    the density exactly: with the option the step's error is that of its FP32 collision, some 30
    roundings of values up to the density (2^-24 each); plain FP32 psi, wrong by 1e-4 between
    neighbours of psi = 0.25, adds 1e-4 * 0.25 / 3 to the force and a sixth of that and more to
    the populations."""
    c = pairs.case(nx, 20, tr=0.8, walls=walls)
    rho = vanishing(c, (20, nx), 3)
    f = np.zeros((9, 20, nx))
    f[0] = rho
    ref = oracle.run(pairs.oracle_params(c), f, 1)
    err = {}
    monkeypatch.setenv("LBM_PERSISTENT", str(persistent))
    for opt in (True, False):
        with pairs.gpu_lattice(c, "fp32", psi_fp64=opt, tile_vec=vec, tile_rows=rows,
                               rho_ref=0.0) as L:
            assert L.persistent == (persistent == 2)
            L.set_populations(f)
            L.step(1)
            err[opt] = np.max(np.abs(L.get_populations() - ref))
    assert err[True] <= 30 * 2.0 ** -24 * rho.max(), err
    assert err[False] > 30 * 2.0 ** -24 * rho.max(), err
