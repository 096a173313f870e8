"""Moments of FP32 fields against extended precision.

Mean: sums of 32 values are exact, the rest are FP64 additions; variance: the
squares are good to 2^-56 of the largest of 32, then the same. The roundings of the
partial sums are random: 4e-16 relative is four units of the last place.
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


def _field(kind, n):
    rng = np.random.default_rng(n)
    z = rng.standard_normal((n, n, n))
    return {"uniform": lambda: rng.random((n, n, n)), "normal": lambda: z, "shifted": lambda: z + 0.3,
            "lognormal": lambda: np.exp(2 * z), "narrow": lambda: 1000 + z, "steps": lambda: 1 + 1e-7 * np.round(z),
            "tiny": lambda: z * 1e-40, "huge": lambda: z * 1e37,
            "mixed": lambda: z * 10.0 ** rng.integers(-30, 8, (n, n, n))}[kind]().astype(np.float32)


@pytest.mark.skipif(np.finfo(np.longdouble).eps > 1e-18, reason="no extended precision on this host")
@pytest.mark.parametrize("n", [32, 54, 96, 162])
@pytest.mark.parametrize("kind", ["uniform", "normal", "shifted", "lognormal", "narrow", "steps", "tiny", "huge",
                                  "mixed"])
def test_mean_and_variance(gg, n, kind):
    f = _field(kind, n)
    x = f.astype(np.longdouble).ravel()
    mean = x.mean()
    var = ((x - mean) ** 2).mean()
    plan = gg.Plan(n, float(n), BBKS, 20.0, "f32")
    got = plan.moments(torch.tensor(f, device="cuda"))
    plan.close()
    assert abs(float((got[1] - var) / var)) < 4e-16
    assert abs(float(got[0] - mean)) < 4e-16 * float(np.abs(x).mean())
    assert got[2] == float(f.min()) and got[3] == float(f.max())
