"""Grid sizes off the tuned list: sizes whose strided tiles take several TMA
boxes of narrow rows (each box must start on a 128-byte boundary of shared
memory), and the size-specialised kernels with one tile shape, against the
oracle and, where the oracle would take minutes, against the FP64 path.

Tolerances as in test_gpu_parity: 1e-5 (FP32) and 1e-12 (FP64) relative L2.
"""
import pytest

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


def check(gg, n, prec):
    plan = gg.Plan(n, float(n), BBKS, 50.0, prec)
    out = plan.zeldovich(seed=5, pos=False)
    plan.sync()
    ora = run_oracle(dict(n=n, box=float(n), cosmo=BBKS, z_init=50.0), seed=5)
    tol = 1e-12 if prec == "f64" else 1e-5
    for k in ("psi", "vel"):
        for j in range(3):
            assert rel_l2(out[k][j].cpu().numpy(), ora[k][j]) < tol, (k, j)
    plan.close()


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_narrow_rows_in_several_boxes(gg, prec):
    check(gg, 324, prec)


@pytest.mark.parametrize("n", [32, 48, 72, 96, 144, 216, 288])
def test_one_shape_sizes_match_oracle(gg, n):
    check(gg, n, "f32")


@pytest.mark.parametrize("n", [432, 576, 648, 768, 864, 1024, 1152])
def test_one_shape_sizes_match_fp64(gg, n):
    ref = gg.Plan(n, float(n), BBKS, 50.0, "f64")
    want = ref.zeldovich(seed=5, pos=False, vel=False)["psi"]
    ref.sync()
    ref.close()
    plan = gg.Plan(n, float(n), BBKS, 50.0, "f32")
    got = plan.zeldovich(seed=5, pos=True, vel=True)
    plan.sync()
    for layout in (False, True):
        plan.set_layout(layout)
        lay = plan.zeldovich(seed=5, psi=False)
        plan.sync()
        for j in range(3):
            assert torch.equal(lay["vel"][j], got["vel"][j]), (layout, j)
            assert torch.equal(lay["pos"][j], got["pos"][j]), (layout, j)
    for j in range(3):
        d = got["psi"][j].double() - want[j]
        assert float(d.norm() / want[j].norm()) < 1e-5, j
    plan.close()
