"""Passes whose launches overlap: calls that follow each other at once, with and
without other kernels between them, give the bits of calls that are waited for
(sizes on both sides of the rule, FP32 and FP64)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BBKS = dict(omega_m=0.3, h=0.7, n_s=0.96, sigma_8=0.8, tf="bbks", omega_l=-1.0,
            omega_b=0.049, t_cmb=2.7255)


@pytest.mark.parametrize("n,prec", [(32, "f32"), (96, "f32"), (256, "f32"), (288, "f32"), (512, "f32"),
                                    (54, "f32"), (162, "f32"), (32, "f64"), (54, "f64"), (64, "f64"), (96, "f64")])
def test_back_to_back_calls(n, prec):
    import paper_2511_10353_gb300 as gg
    plan = gg.Plan(n, float(n), BBKS, 50.0, prec)
    single = {}
    for seed in (1, 2, 3):
        single[seed] = plan.zeldovich(seed=seed)["pos"]
        plan.sync()
    for between in (False, True):
        rows = []
        for seed in (1, 2, 3, 1, 2, 3):
            out = plan.zeldovich(seed=seed)["pos"]
            rows.append((seed, [o * 1 for o in out] if between else out))
        plan.sync()
        for seed, out in rows:
            for j in range(3):
                assert torch.equal(out[j], single[seed][j]), (seed, j, between)
