"""The adjoint's two-input passes and the cloud-in-cell walk at the edges of
their shapes.

The transpose of all three displacements at once (joined spectra) against the
sum of the single-component chains: two FP32 chains of 4e-7 relative L2 each
leave 2e-6, FP64 ones of 2e-15 leave 1e-14. Density and its adjoint against
the oracle on scattered, coherent and exactly nodal displacements: an FP32
coordinate u is off by up to u 2^-24 per axis, and each cell sums the weights
of a few particles, so |u| < 2 N (N <= 54) stays within 1e-4 relative L2;
FP64 within 1e-12.
"""
import numpy as np
import pytest

from oracle import adjoint as oadj

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


@pytest.mark.parametrize("n,prec", [(n, "f32") for n in (32, 48, 64, 72, 96, 128, 144, 192, 216, 256, 288,
                                                         384, 432, 512, 576, 648, 768)]
                         + [(64, "f64"), (512, "f64"), (40 + 8, "f64")])
def test_joined_transpose_is_the_sum(gg, n, prec):
    dt = torch.float64 if prec == "f64" else torch.float32
    plan = gg.Plan(n, float(n), BBKS, 20.0, prec)
    gen = torch.Generator(device="cuda").manual_seed(n)
    g = [torch.randn((n, n, n), dtype=dt, device="cuda", generator=gen) for _ in range(3)]
    got = plan.zeldovich_adjoint(g)
    want = sum(plan.zeldovich_adjoint([g[j] if i == j else None for i in range(3)]).double()
               for j in range(3))
    plan.sync()
    plan.close()
    assert float((got.double() - want).norm() / want.norm()) < (2e-6 if prec == "f32" else 1e-14)


def _displacements(kind, n, cell, rng):
    if kind == "scattered":  # neighbours far apart, some beyond the box
        return [rng.uniform(-1.0, 1.0, (n, n, n)) * n * cell for _ in range(3)]
    if kind == "nodal":      # every particle on a node, whole cells away
        return [cell * rng.integers(-2, 3, (n, n, n)).astype(float) for _ in range(3)]
    i = np.arange(n) * 2 * np.pi / n  # coherent: neighbours share nodes
    s = np.sin(i)[:, None, None] + np.cos(i)[None, :, None] + np.sin(2 * i)[None, None, :]
    return [cell * (0.3 * s + 0.05 * rng.standard_normal((n, n, n))) for _ in range(3)]


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("kind", ["coherent", "scattered", "nodal"])
@pytest.mark.parametrize("n", [6, 32, 36, 54])
def test_cic_walk(gg, n, kind, prec):
    dt = torch.float64 if prec == "f64" else torch.float32
    box = 1.5 * n
    rng = np.random.default_rng(n)
    psi = [torch.tensor(v, dtype=dt, device="cuda") for v in _displacements(kind, n, box / n, rng)]
    gd = torch.tensor(rng.standard_normal((n, n, n)), dtype=dt, device="cuda")
    plan = gg.Plan(n, box, BBKS, 20.0, prec)
    delta = plan.cic_density(psi)
    gp = plan.cic_density_adjoint(psi, gd)
    plan.sync()
    plan.close()
    host = [p.cpu().numpy().astype(np.float64) for p in psi]
    tol = 1e-12 if prec == "f64" else 1e-4
    want = oadj.cic_density(host, box)
    d = delta.cpu().numpy() - want
    assert np.linalg.norm(d) <= tol * (np.linalg.norm(want) + n ** 1.5)
    if kind == "nodal" and prec == "f32":
        return  # one-sided on a node plane: an FP32 rounding picks the side
    wa = oadj.cic_adjoint(host, gd.cpu().numpy().astype(np.float64), box)
    clear = np.ones((n, n, n), dtype=bool)
    if prec == "f32":  # the derivative jumps at node planes: leave out who rounds across one
        for j in range(3):
            sh = [1, 1, 1]
            sh[j] = n
            u = np.arange(n).reshape(sh) + host[j] * n / box
            clear &= np.abs(u - np.round(u)) > 2.0 ** -22 * (np.abs(u) + 1)
    for j in range(3):
        diff = np.where(clear, gp[j].cpu().numpy() - wa[j], 0.0)
        assert np.linalg.norm(diff) <= tol * 10 * np.linalg.norm(wa[j])
