"""The fixed-point FP64 transforms at the large grids, and of extreme values.

Accuracy: smoothing with radius 0 runs the six transforms forward and back and
is the identity but for the |m_j| = N/2 modes, which alternating sums take out of
the input. Rounding a flat column of N to its unit (at most sum |z| 2^-61.5)
changes the outputs by 0.41 N 2^-61.5 relative rms at most, the products of the
first stages bring that to 1.3 times: 2.3e-16 at N = 1536. Four strided
transforms, two along z of half the length and six roundings to FP64 stay below
5.5e-16 in quadrature; the bound is 6e-16. (FP64 floating-point transforms:
5.7e-16 at 512 to 6.6e-16 at 1536.)
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


def _white(n):
    f = torch.empty((n, n, n), dtype=torch.float64, device="cuda")
    for i in range(n):
        f[i].normal_(generator=torch.Generator(device="cuda").manual_seed(i))
    return f


@pytest.mark.parametrize("n", [384, 512, 768, 1024, 1536])
def test_forward_and_back(gg, n):
    plan = gg.Plan(n, float(n), BBKS, 50.0, "f64")
    f = _white(n)
    out = torch.empty_like(f)
    sign = 1.0 - 2.0 * (torch.arange(n, device="cuda", dtype=torch.float64) % 2)
    for scale in (1.0, 1.18, 1.2, 1.19):  # the block scale steps in powers of two: 1, 1.18, 1.42, 1.69
        f.mul_(scale)
        plan.smooth(f, 0.0, out=out)
        plan.sync()
        mx = sum(f[i] * float(sign[i]) for i in range(n)) / n
        num = den = 0.0
        for i in range(0, n, n // 64):
            w = f[i] - float(sign[i]) * mx
            w = w - sign[:, None] * (sign[:, None] * w).mean(0)[None, :]
            w = w - sign[None, :] * (sign[None, :] * w).mean(1)[:, None]
            num += float(((out[i] - w) ** 2).sum())
            den += float((w ** 2).sum())
        assert (num / den) ** 0.5 < 6e-16, scale
    plan.close()
    del f, out
    torch.cuda.empty_cache()


@pytest.mark.parametrize("n", [96, 192, 384, 512, 768, 1024, 1536])
def test_no_systematic_rounding(gg, n):
    """Errors of one sign add up in single modes and cells: the modes along the axes
    keep the bound of the whole field, and no cell is off by more than 12 times the
    rms error (normal errors: 6.3 times among 1536^3)."""
    plan = gg.Plan(n, float(n), BBKS, 50.0, "f64")
    f = _white(n)
    out = plan.smooth(f, 0.0)
    plan.sync()
    plan.close()
    sign = 1.0 - 2.0 * (torch.arange(n, device="cuda", dtype=torch.float64) % 2)
    mx = sum(f[i] * float(sign[i]) for i in range(n)) / n
    err = [torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(3)]
    ref = [torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(3)]
    num = worst = 0.0
    for i in range(n):
        w = f[i] - float(sign[i]) * mx
        w = w - sign[:, None] * (sign[:, None] * w).mean(0)[None, :]
        w = w - sign[None, :] * (sign[None, :] * w).mean(1)[:, None]
        d = out[i] - w
        num += float((d ** 2).sum())
        worst = max(worst, float(d.abs().max()))
        for s, v in ((err, d), (ref, w)):
            s[0][i] = v.sum()
            s[1] += v.sum(1)
            s[2] += v.sum(0)
    assert worst < 12 * (num / n ** 3) ** 0.5
    for e, r in zip(err, ref):
        assert float((e - e.mean()).norm() / (r - r.mean()).norm()) < 6e-16
    del f, out
    torch.cuda.empty_cache()


@pytest.mark.parametrize("n", [768, 1024])
def test_displacement_against_fft(gg, n):
    """psi of caller noise against FP64 transforms of another library, 1e-12."""
    box = float(n)
    f = _white(n)
    plan = gg.Plan(n, box, BBKS, 50.0, "f64")
    psi = plan.zeldovich(noise=f, pos=False, vel=False)["psi"]
    plan.sync()
    plan.close()
    q = 3 * (n // 2) ** 2 + 1
    u = gg.filter_table(n, box, BBKS, 50.0, q) / n ** 1.5 * (box / (2 * np.pi))
    u[1:] /= np.arange(1, q)
    u = torch.tensor(u, device="cuda")
    spec = torch.fft.rfftn(f)
    del f
    m = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64).round()
    mz = torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64)
    keep = [m != -n // 2, m != -n // 2, mz != n // 2]
    for i in range(n):
        m2 = (m[i] ** 2 + m[:, None] ** 2 + mz[None, :] ** 2).long()
        ok = keep[0][i] & keep[1][:, None] & keep[2][None, :]
        spec[i] *= torch.where(ok, u[m2.clamp(max=q - 1)], 0.0)
    for j, mj in enumerate((m[:, None, None], m[None, :, None], mz[None, None, :])):
        want = torch.fft.irfftn(1j * mj * spec, s=(n, n, n), norm="forward")
        want.sub_(psi[j])
        assert float(want.norm() / psi[j].norm()) < 1e-12, j
        del want
        torch.cuda.empty_cache()


@pytest.mark.parametrize("n", [32, 72, 96, 256])
def test_dominated_column(gg, n):
    """Beside one value of 1e6 the rest of a field keeps its absolute accuracy: three
    results, each within 6e-16 of the dominating one's norm."""
    plan = gg.Plan(n, float(n), BBKS, 50.0, "f64")
    f = torch.randn((n, n, n), dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(n))
    f[0, 0, 0] = 0.0
    spike = torch.zeros_like(f)
    spike[0, 0, 0] = 1e6
    one, ref, got = (plan.gaussian_field(noise=x) for x in (spike, f, f + spike))
    plan.sync()
    plan.close()
    tol = 1.8e-15 * float(one.norm())
    assert tol < 1e-6 * float(ref.norm())  # the check sees the rest of the field
    assert float((got - one - ref).norm()) < tol


@pytest.mark.parametrize("n", [32, 64, 96])
def test_subnormal_field(gg, n):
    """A field of subnormal values, forward and back. After the factor 1 / n^3 the
    spectrum is rounded to multiples of 2^-1074; n^3 such roundings of rms 0.3 (more on
    the way back, growing less) add up to 0.5 n^1.5 units rms, 8 times that at most."""
    plan = gg.Plan(n, float(n), BBKS, 50.0, "f64")
    f = torch.ldexp(_white(n), torch.tensor(-1032.0, device="cuda", dtype=torch.float64))
    assert 0 < float(f.abs().max()) < 2.0 ** -1022
    got = plan.smooth(f, 0.0)
    plan.sync()
    plan.close()
    up = lambda x: torch.ldexp(x, torch.tensor(1000.0, device="cuda", dtype=torch.float64))
    w = up(f)
    for axis in range(3):  # the |m_j| = N/2 modes, dropped
        s = (1.0 - 2.0 * (torch.arange(n, device="cuda", dtype=torch.float64) % 2)).reshape(
            [-1 if a == axis else 1 for a in range(3)])
        w = w - s * (s * w).mean(axis, keepdim=True)
    assert float((up(got) - w).abs().max()) < 8 * 0.5 * n ** 1.5 * 2.0 ** -74
