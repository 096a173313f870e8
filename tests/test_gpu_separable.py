"""Separable filters (Gaussian smoothing, degrading) as one pass per axis, FP32,
against the oracle at sizes of every schedule shape, and the run-time sizes that
keep the chain. Two FP32 transforms and a filter: 1e-6 relative L2 is three
times what the other FP32 paths show, the bound of the parity tests is 1e-5.
"""
import numpy as np
import pytest

from oracle import adjoint as oadj, particles as opart

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BBKS = dict(omega_m=0.3, h=0.7, n_s=0.96, sigma_8=0.8, tf="bbks", omega_l=-1.0,
            omega_b=0.049, t_cmb=2.7255)
SIZES = [32, 36, 48, 64, 72, 96, 128, 144, 162, 192, 216, 256, 288, 384]


@pytest.fixture(scope="module")
def gg():
    from paper_2511_10353_gb300 import build
    build.build(verbose=False)
    import paper_2511_10353_gb300 as m
    return m


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("n", SIZES)
def test_smooth(gg, n):
    f = np.random.default_rng(n).standard_normal((n, n, n)).astype(np.float32)
    plan = gg.Plan(n, 2.0 * n, BBKS, 20.0, "f32")
    for radius in (3.0, 9.0, 0.0):  # the table changes with the radius
        t = torch.tensor(f, device="cuda")
        got = plan.smooth(t, radius)
        plan.smooth(t, radius, out=t)
        plan.sync()
        assert torch.equal(got, t)
        assert _rel(got.cpu().numpy(), oadj.smooth(f.astype(np.float64), 2.0 * n, radius)) < 1e-5
    plan.close()


@pytest.mark.parametrize("n,r", [(n, 2) for n in SIZES if n <= 192] + [(72, 3), (64, 5), (48, 4), (96, 1)])
def test_degrade(gg, n, r):
    f = np.random.default_rng(n).standard_normal((n * r, n * r, n * r)).astype(np.float32)
    plan = gg.Plan(n, 50.0, BBKS, 20.0, "f32")
    got = plan.degrade(torch.tensor(f, device="cuda"))
    plan.sync()
    plan.close()
    assert _rel(got.cpu().numpy(), opart.degrade(f, r)) < 1e-5
