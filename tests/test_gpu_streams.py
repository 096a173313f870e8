"""Calls that follow each other on a side stream without a synchronisation, and
distinct plans on several host threads: results equal those of lone calls.
"""
import threading

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


@pytest.mark.parametrize("n,prec", [(256, "f32"), (162, "f32"), (128, "f64")])
def test_smoothing_radii_back_to_back(gg, n, prec):
    """The filter table of one radius stays while passes of that radius run."""
    dt = torch.float32 if prec == "f32" else torch.float64
    f = torch.randn((n, n, n), dtype=dt, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    plan = gg.Plan(n, 2.0 * n, BBKS, 20.0, prec)
    radii = (3.0, 9.0, 5.0)
    want = []
    for r in radii:
        want.append(plan.smooth(f, r))
        plan.sync()
    torch.cuda.synchronize()
    reps = 24  # queued work of one radius when the next one's table is written
    got = [torch.empty_like(f) for _ in range(reps * len(radii))]
    with torch.cuda.stream(torch.cuda.Stream()):
        for i, r in enumerate(radii):
            for q in range(reps):
                plan.smooth(f, r, out=got[i * reps + q])
        plan.sync()
    torch.cuda.synchronize()
    for i in range(len(radii)):
        for q in range(reps):
            assert torch.equal(got[i * reps + q], want[i]), (radii[i], q)
    plan.close()


def test_merges_on_two_threads(gg):
    """Coarse grids of different sizes need different shared memory in one kernel."""
    n, box, runs = 512, 500.0, 150
    errors = []

    def work(nl, seed):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                plan = gg.Plan(n, box, BBKS, 20.0, "f32")
                large = [torch.full((nl, nl, nl), 0.01, device="cuda") for _ in range(3)]
                out = {"psi": [plan.empty() for _ in range(3)], "pos": [None] * 3, "vel": [None] * 3}
                for _ in range(runs):
                    plan.zeldovich_merge(large, 2 * box / nl, seed=seed, out=out)
                plan.sync()
                plan.close()
        except Exception as e:  # reported by the test's thread
            errors.append((nl, repr(e)))

    threads = [threading.Thread(target=work, args=(nl, i)) for i, nl in enumerate((256, 128))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
