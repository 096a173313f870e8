"""FP64 autotuning: the faster of the two spectrum layouts, timed, not guessed;
results are bit-identical whatever it takes.
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


def _time(plan, out, reps=5):
    plan.zeldovich(seed=1, out=out)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    for _ in range(reps):
        plan.zeldovich(seed=1, out=out)
    b.record()
    b.synchronize()
    return a.elapsed_time(b) / reps


@pytest.mark.parametrize("n", [64, 512, 768])
def test_layout(gg, n):
    plan = gg.Plan(n, float(n), BBKS, 50.0, "f64")
    out = {"psi": [None] * 3, "pos": [plan.empty() for _ in range(3)], "vel": [plan.empty() for _ in range(3)]}
    ms = []
    for chunked in (False, True):
        plan.set_layout(chunked)
        ms.append(_time(plan, out))
    print("n %d: plain %.3f ms, chunk-major %.3f ms" % (n, *ms))
    ref = [t.clone() for t in out["pos"] + out["vel"]]
    for start in (False, True):
        plan.set_layout(start)
        plan.autotune(3)
        # a run at 64^3 lasts as long as its launches: no timing decides there
        if n > 64 and abs(ms[1] - ms[0]) > 0.03 * ms[0]:  # else either may win
            assert plan.layout() == (ms[1] < ms[0]), ms
        plan.zeldovich(seed=1, out=out)
        plan.sync()
        for a, b in zip(out["pos"] + out["vel"], ref):
            assert torch.equal(a, b)
    plan.close()
