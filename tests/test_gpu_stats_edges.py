"""The diagnostics at the edges of their kernels: shell orbits of the smallest
and of odd-half grids, and fields that the FP32 moments cannot add as integers
(wide ranges, a large mean, infinities, NaN, tiny values, unaligned views).

The moments are compared with FP64 numpy: sums of M values of size s carry at
most M s 2^-53 in either order, so mean and variance agree to 1e-13 of the
mean absolute (squared) value, plus for the variance the rounding of the mean.
"""
import numpy as np
import pytest

from oracle import stats as ostats

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BBKS = dict(omega_m=0.3, h=0.7, n_s=0.96, sigma_8=0.8, tf="bbks", omega_l=-1.0,
            omega_b=0.049, t_cmb=2.7255)


@pytest.fixture(scope="module")
def gg():
    from paper_2511_10353_gb300 import build
    build.build(verbose=False)
    import paper_2511_10353_gb300 as m
    return m


@pytest.mark.parametrize("n,prec", [(4, "f64"), (6, "f32"), (18, "f64"), (54, "f32"), (72, "f32"), (96, "f64")])
def test_shells(gg, n, prec):
    rng = np.random.default_rng(n)
    f = rng.standard_normal((n, n, n))
    plan = gg.Plan(n, 2.0 * n, BBKS, 20.0, prec)
    dt = torch.float64 if prec == "f64" else torch.float32
    k, p, c = plan.power_spectrum(torch.tensor(f, dtype=dt, device="cuda"))
    plan.close()
    kw, pw, cw = ostats.power_spectrum(f, 2.0 * n, n // 2)
    tol = 1e-12 if prec == "f64" else 1e-5
    assert np.array_equal(c, cw)
    assert np.abs(k - kw).max() <= 1e-12 * kw.max()
    # the k = 0 shell is one mode: its error is that of the sum over the field
    assert np.all(np.abs(p - pw) <= tol * (np.abs(pw) + pw.mean()))


def _fields(kind, n, rng):
    f = rng.standard_normal(n ** 3).astype(np.float32)
    if kind == "wide":
        f *= np.exp(rng.uniform(-40, 40, n ** 3)).astype(np.float32)
    elif kind == "mean":
        f = (f + np.float32(1.0e5)).astype(np.float32)
    elif kind == "tiny":
        f *= np.float32(1e-30)
    elif kind == "denormal":
        f *= np.float32(1e-41)
    elif kind == "huge":
        f *= np.float32(1e30)
    elif kind == "zero":
        f[:] = 0
    return f


@pytest.mark.parametrize("kind", ["plain", "wide", "mean", "tiny", "denormal", "huge", "zero"])
@pytest.mark.parametrize("n", [6, 48, 96])
def test_moments(gg, kind, n):
    f = _fields(kind, n, np.random.default_rng(n))
    plan = gg.Plan(n, 10.0, BBKS, 20.0, "f32")
    mean, var, lo, hi = plan.moments(torch.tensor(f, device="cuda").reshape(n, n, n))
    plan.close()
    d = f.astype(np.float64)
    m = d.mean()
    assert abs(mean - m) <= 1e-13 * np.abs(d).mean()
    want = np.mean((d - m) ** 2)
    assert abs(var - want) <= 1e-13 * want + (1e-13 * np.abs(d).mean()) ** 2
    assert lo == d.min() and hi == d.max()


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_moments_not_finite(gg, bad):
    n = 48
    f = np.random.default_rng(1).standard_normal(n ** 3).astype(np.float32)
    f[777] = bad
    plan = gg.Plan(n, 10.0, BBKS, 20.0, "f32")
    mean, var, lo, hi = plan.moments(torch.tensor(f, device="cuda").reshape(n, n, n))
    plan.close()
    with np.errstate(invalid="ignore"):
        want = f.astype(np.float64).mean()
    assert (np.isnan(mean) and np.isnan(want)) or mean == want
    assert np.isnan(var)
    finite = f[np.isfinite(f)]
    assert lo == (bad if bad == -np.inf else finite.min()) and hi == (bad if bad == np.inf else finite.max())


def test_moments_unaligned_view(gg):
    n = 48
    base = torch.randn(n ** 3 + 1, device="cuda")
    f = base[1:].reshape(n, n, n)
    plan = gg.Plan(n, 10.0, BBKS, 20.0, "f32")
    mean, var, lo, hi = plan.moments(f)
    plan.close()
    d = f.cpu().numpy().astype(np.float64)
    assert abs(mean - d.mean()) <= 1e-13 and abs(var - d.var()) <= 1e-13 * d.var()
    assert lo == d.min() and hi == d.max()
