"""The fixed-point transforms of the FP64 path: every specialised size against
the oracle, accuracy against extended precision, powers of two as scales (the
block exponents must make them exact), zeros, infinities and NaN.

Accuracy: six transforms, each within 2^-53 (see the bound of the block scale),
six roundings to FP64 and one of the filter: in quadrature below 4e-16.
"""
import numpy as np
import pytest
import scipy.fft as sfft

from tests.gpu_helpers import rel_l2, run_oracle

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


@pytest.mark.parametrize("n", [32, 48, 64, 72, 96, 128, 144, 192, 216, 256, 288])
def test_sizes_match_oracle(gg, n):
    plan = gg.Plan(n, float(n), BBKS, 50.0, "f64")
    out = plan.zeldovich(seed=5)
    ora = run_oracle(dict(n=n, box=float(n), cosmo=BBKS, z_init=50.0), seed=5)
    for j in range(3):
        for k in ("psi", "vel"):
            assert rel_l2(out[k][j].cpu().numpy(), ora[k][j]) < 1e-12, (k, j)
    plan.set_layout(True)  # chunk-major spectra
    lay = plan.zeldovich(seed=5)
    plan.sync()
    for j in range(3):
        assert torch.equal(lay["pos"][j], out["pos"][j]), j
    plan.close()


@pytest.mark.skipif(np.finfo(np.longdouble).eps > 1e-18, reason="no extended precision on this host")
@pytest.mark.parametrize("n", [48, 64, 96])
@pytest.mark.parametrize("kind", ["white", "steep", "spike"])
def test_accuracy(gg, n, kind):
    rng = np.random.default_rng(n)
    f = rng.standard_normal((n, n, n))
    m = np.fft.fftfreq(n, 1 / n).round().astype(np.int64)
    m2 = m[:, None, None] ** 2 + m[None, :, None] ** 2 + np.arange(n // 2 + 1)[None, None, :] ** 2
    if kind == "steep":
        f = np.fft.irfftn(np.fft.rfftn(f) / (1.0 + m2) ** 2, s=f.shape, axes=(0, 1, 2))
    elif kind == "spike":
        f = np.zeros((n, n, n))
        f[1, n // 2, 7], f[0, 0, 0] = 1.0, 1e-3
    plan = gg.Plan(n, float(n), BBKS, 50.0, "f64")
    got = plan.gaussian_field(noise=torch.tensor(f, device="cuda"))
    plan.sync()
    plan.close()
    s = gg.filter_table(n, float(n), BBKS, 50.0, 3 * (n // 2) ** 2 + 1) * (1.0 / float(n) ** 1.5)
    keep = (m[:, None, None] != -n // 2) & (m[None, :, None] != -n // 2) & (np.arange(n // 2 + 1) != n // 2)
    spec = sfft.rfftn(f.astype(np.longdouble)) * np.where(keep, s[m2], 0.0).astype(np.longdouble)
    want = sfft.irfftn(spec, s=f.shape, axes=(0, 1, 2), norm="forward")
    d = got.cpu().numpy().astype(np.longdouble) - want
    assert float(np.sqrt((d * d).sum() / (want * want).sum())) < 4e-16


@pytest.mark.parametrize("n", [32, 72, 96])
def test_scales(gg, n):
    plan = gg.Plan(n, float(n), BBKS, 50.0, "f64")
    f = torch.randn((n, n, n), dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(n))
    ref = plan.gaussian_field(noise=f)
    for e in (-900, -400, 400, 850):
        got = plan.gaussian_field(noise=torch.ldexp(f, torch.tensor(e, device="cuda")))
        back = torch.ldexp(got, torch.tensor(-e, device="cuda"))
        assert torch.equal(back, ref), e
    assert float(plan.gaussian_field(noise=torch.zeros_like(f)).abs().max()) == 0.0
    wide = f.clone()
    wide[0, 0, 0] = 1e30  # one value dominates every line and column
    got = plan.gaussian_field(noise=wide)
    one = plan.gaussian_field(noise=torch.where(wide == 1e30, wide, 0.0))
    assert float((got - one - ref).norm()) < 1e-12 * float(one.norm())
    for bad in (float("inf"), float("nan")):
        wide[1, 2, 3] = bad
        assert bool(plan.gaussian_field(noise=wide).isnan().all())
    plan.sync()
    plan.close()
