"""Margins of the lazy evaluation vs the reference decoder, bit for bit, where the rounding of E_k
is as wide as the noise: samples and thresholds of the same size, far above the margin's step.
"""
import numpy as np
import pytest

from paper_1402_2773_gb300 import ngdbf, workload as wl
from test_gpu_parity import O, _gpu, assert_parity  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [dict(), dict(precision=ngdbf.NGDBF_FP16)], ids=["fp32", "fp16"])
@pytest.mark.parametrize("variant", [0, 1, 2, 3, 3 | 8])
@pytest.mark.parametrize("theta", [1.0, 64.0, 2048.0])
def test_samples_at_a_large_threshold(O, theta, variant, prec):
    """Unsaturated samples on both sides of a positive threshold at a power of two, where the
    spacing of the held values doubles: rounding x_k y_k + w S_k moves E_k by half a spacing, up to
    three standard deviations of the noise here."""
    code = wl.peg_code(504, 252, 3, seed=3)
    ulp = theta * 2.0 ** -10                              # binary16 spacing above theta
    rng = np.random.default_rng(7)
    y = theta + rng.choice([-0.5, 0.0, 1.0], size=(64, code.n)) * ulp
    y = (y * rng.choice([1.0, -1.0], size=y.shape, p=[0.9, 0.1])).astype(np.float32)
    assert_parity(O, code, y, 0.32 * ulp, seed=5, variant=variant, lam=0.999, t_max=12, smooth_window=4,
                  w=0.165 * ulp, theta=theta, eta=0.5, y_max=0.0, **prec)


@pytest.mark.parametrize("prec", [dict(), dict(precision=ngdbf.NGDBF_FP16)], ids=["fp32", "fp16"])
@pytest.mark.parametrize("variant", [0, 3, 4, 6])
@pytest.mark.parametrize("y_max", [0.0, 2.5])
def test_samples_that_are_not_numbers(O, variant, y_max, prec):
    """Such a symbol's E_k is evaluated in every iteration and never below a threshold, nor the least of
    a frame (the single-bit variant; not symbol 0, where the reference decoder starts its search)."""
    code = wl.peg_code(504, 252, 3, seed=3)
    y, _, sig = wl.frames(code, 64, 3.0, seed=9)
    rng = np.random.default_rng(4)
    at = rng.random(y.shape)
    at[:, 0] = 1.0
    y[at < 0.02] = np.nan
    y[(at >= 0.02) & (at < 0.025)] = -np.inf
    assert_parity(O, code, y, sig, seed=6, variant=variant, lam=0.97, t_max=30, smooth_window=10, y_max=y_max, **prec)
