"""The layout switch on a plan as it was made: chunk-major takes effect at every
size with specialised kernels, results are bit-identical, and switching back
restores the default tile variants; variants that were set are left alone.
"""
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


@pytest.mark.parametrize("n,prec", [(64, "f32"), (192, "f32"), (256, "f32"), (384, "f32"), (512, "f32"),
                                    (576, "f32"), (128, "f64"), (384, "f64")])
def test_switch_takes_effect(gg, n, prec):
    plan = gg.Plan(n, float(n), BBKS, 50.0, prec)
    default = plan.variants()
    out = []
    for chunked in (False, True):
        plan.set_layout(chunked)
        assert plan.layout() is chunked
        out.append(plan.zeldovich(seed=4))
        plan.sync()
    for k in ("psi", "pos", "vel"):
        for j in range(3):
            assert torch.equal(out[0][k][j], out[1][k][j]), (k, j)
    plan.set_layout(False)
    assert plan.variants() == default
    plan.close()


def test_set_variants_are_kept(gg):
    plan = gg.Plan(512, 512.0, BBKS, 50.0, "f32")
    mixed = [0, 0, 2, 0, 1, 0]  # tile widths differ
    plan.set_variants(mixed)
    plan.set_layout(True)
    assert plan.variants() == mixed and not plan.layout()
    plan.close()
