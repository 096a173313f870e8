"""The merge's coarse lines staged in shared memory (FP32, specialised sizes)
against the general interpolation (FP64 reads the coarse grid itself) over grid
ratios that divide and that do not, one coarse cell and equal grids; positions
and velocities alone (a kernel of their own); and infinities and NaN, which reach
exactly the fine cells whose interpolation reads them.

Tolerances: 1e-5 relative L2, the FP32 bound of the parity tests; positions four
units in the last place of L besides.
"""
import numpy as np
import pytest

from tests.gpu_helpers import min_image

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BBKS = dict(omega_m=0.3, h=0.7, n_s=0.96, sigma_8=0.8, tf="bbks", omega_l=-1.0,
            omega_b=0.049, t_cmb=2.7255)
RATIOS = [(64, 32), (96, 72), (72, 72), (64, 1), (48, 2), (96, 64), (128, 54), (256, 128)]


@pytest.fixture(scope="module")
def gg():
    from paper_2511_10353_gb300 import build
    build.build(verbose=False)
    import paper_2511_10353_gb300 as m
    return m


def _large(nl):
    rng = torch.Generator(device="cuda").manual_seed(nl)
    return [torch.randn((nl, nl, nl), generator=rng, device="cuda", dtype=torch.float64) for _ in range(3)]


@pytest.mark.parametrize("psi", [True, False])
@pytest.mark.parametrize("nh,nl", RATIOS)
def test_against_fp64(gg, nh, nl, psi):
    box = 2.0 * nh
    large, out = _large(nl), {}
    for prec, dt in (("f64", torch.float64), ("f32", torch.float32)):
        plan = gg.Plan(nh, box, BBKS, 30.0, prec)
        out[prec] = plan.zeldovich_merge([g.to(dt) for g in large], 2 * box / nl, seed=3, psi=psi or prec == "f64")
        plan.sync()
        plan.close()
    ulp = float(np.spacing(np.float32(box)))
    for j in range(3):
        for k in ("psi", "vel") if psi else ("vel",):
            a, b = out["f32"][k][j].double(), out["f64"][k][j]
            assert float((a - b).norm() / b.norm()) < 1e-5, (k, j)
        d = min_image((out["f32"]["pos"][j].double() - out["f64"]["pos"][j]).cpu().numpy(), box)
        assert np.abs(d).max() < 4 * ulp + 1e-5 * float(out["f64"]["psi"][j].abs().max()), j


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
@pytest.mark.parametrize("nh,nl", RATIOS)
def test_nonfinite_coarse_cell(gg, nh, nl, bad):
    box, cell = 2.0 * nh, (nl // 2, nl // 3, nl - 1)
    plan = gg.Plan(nh, box, BBKS, 30.0, "f32")
    large = [g.float() for g in _large(nl)]
    for g in large:
        g[cell] = bad
    out = plan.zeldovich_merge(large, 2 * box / nl, seed=3, pos=False)
    plan.sync()
    plan.close()
    i0 = ((2 * np.arange(nh) + 1) * nl - nh) // (2 * nh)  # coarse cell centre below each fine one
    reads = [(i0 % nl == c) | ((i0 + 1) % nl == c) for c in cell]
    want = reads[0][:, None, None] & reads[1][None, :, None] & reads[2][None, None, :]
    for j in range(3):
        for k in ("psi", "vel"):
            assert np.array_equal(~np.isfinite(out[k][j].cpu().numpy()), want), (k, j)
