"""FP64 white noise, every value against extended precision in units of its own
last place, small values included.

Bound: the logarithm is within 0.7 units, the root within 0.9 of its exact value
then, sine and cosine within 1.6, the product adds 0.5: below 4 units where the
unit is the smallest a value of that size can have.
"""
import numpy as np
import pytest

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


@pytest.mark.skipif(np.finfo(np.longdouble).eps > 1e-18, reason="no extended precision on this host")
@pytest.mark.parametrize("seed", [1, 2])
def test_every_value(gg, seed):
    ld = np.longdouble
    n = 96
    words = gg.noise_bits(seed, 0, n ** 3 // 4).cpu().numpy().view(np.uint32).astype(np.int64).reshape(-1, 2)
    plan = gg.Plan(n, float(n), BBKS, 50.0, "f64")
    got = plan.white_noise(seed).cpu().numpy().reshape(-1, 2)
    plan.sync()
    plan.close()
    two32 = ld(2) ** 32
    # -log(1 - v) near u = 1 by its own series in log1p
    rho = np.sqrt(-2 * np.log1p(-(ld(2 ** 32 - 1) - words[:, 0].astype(ld)) / two32))
    quarter = (words[:, 1] + (1 << 29)) >> 30  # the angle reduced by integers: no digits lost near an axis
    x = ld("6.283185307179586476925286766559005768") * ((words[:, 1] - (quarter << 30)).astype(ld) / two32)
    s, c, q = np.sin(x), np.cos(x), quarter % 4
    want = np.stack([rho * np.choose(q, [c, -s, -c, s]), rho * np.choose(q, [s, c, -s, -c])], 1)
    assert np.all(got[want == 0] == 0)
    ok = want != 0
    ulp = np.spacing(np.abs(want[ok]).astype(np.float64)).astype(ld)
    err = np.abs(got[ok].astype(ld) - want[ok]) / ulp
    assert float(err.max()) < 4.0
    assert float(np.sqrt(((got.astype(ld) - want) ** 2).sum() / (want ** 2).sum())) < 8.4e-17
