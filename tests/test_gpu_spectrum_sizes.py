"""P(k) of FP32 fields at sizes with several tile shapes against the FP64 path
(at N = 384 its strided passes run the general radices, not the other passes').

FP32 transforms of white noise are off by about 3e-7 a mode, independently; a
shell has 18 modes or more: below 2e-7 of P(k), bound 1e-6 of its largest value.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BBKS = dict(omega_m=0.3, h=0.7, n_s=0.96, sigma_8=0.8, tf="bbks", omega_l=-1.0,
            omega_b=0.049, t_cmb=2.7255)


@pytest.mark.parametrize("n", [192, 256, 384])
def test_power_spectrum_against_fp64(n):
    import paper_2511_10353_gb300 as gg
    p32 = gg.Plan(n, float(n), BBKS, 50.0, "f32")
    p64 = gg.Plan(n, float(n), BBKS, 50.0, "f64")
    w = p32.white_noise(seed=9)
    _, p, c = p32.power_spectrum(w)
    _, p2, c2 = p64.power_spectrum(w.double())
    assert np.array_equal(c, c2)
    assert np.max(np.abs(p - p2)) < 1e-6 * np.max(p2)
