"""Lazy evaluation of E_k (only outputs at or below a margin's cutoff are evaluated) vs the reference
decoder, bit for bit, where its quantization is under strain: weights, thresholds, noise scales and
sample ranges far apart, every symbol degree up to the 4-bit counts' limit and the bit-sliced counts
above it, non-finite samples, and every number of live slots.
"""
import gc

import numpy as np
import pytest

import oracle
from paper_1402_2773_gb300 import ngdbf, workload as wl
from test_gpu_parity import O, _gpu, assert_parity  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _collect():
    """Tensors held by reference cycles of earlier tests go now, not while a later test counts memory."""
    yield
    gc.collect()


def code_with_degree(n, m, top, seed):
    """Random H, symbol degrees 2..4 and one symbol of degree `top` in every 16."""
    rng = np.random.default_rng(seed)
    H = np.zeros((m, n), np.uint8)
    for k in range(n):
        H[rng.choice(m, size=top if k % 16 == 5 else int(rng.integers(2, 5)), replace=False), k] = 1
    for i in np.nonzero(H.sum(1) == 0)[0]:
        H[i, rng.integers(n)] = 1
    return wl.code_from_dense(H)


PREC = [dict(), dict(precision=ngdbf.NGDBF_FP16), dict(precision=ngdbf.NGDBF_FIX, q_bits=3),
        dict(precision=ngdbf.NGDBF_FIXACC, q_bits=8)]


@pytest.mark.parametrize("top", [7, 8, 15, 16, 20])
@pytest.mark.parametrize("variant", [0, 1, 3, 4, 6, 3 | 8])
def test_degrees(O, top, variant):
    code = code_with_degree(150, 80, top, seed=top)
    y, _, _ = wl.frames(code, 45, None, seed=7, sigma=0.6)
    for prec in PREC:
        assert_parity(O, code, y, 0.6, seed=3, variant=variant, lam=0.97, t_max=25, smooth_window=6, w=0.3,
                      theta=-0.6, **prec)


@pytest.mark.parametrize("variant", [0, 3, 6, 3 | 8])
@pytest.mark.parametrize("kw", [
    dict(w=1e-3), dict(w=20.0), dict(theta=0.4), dict(theta=-30.0, w=9.0), dict(eta=0.0), dict(eta=1e-3),
    dict(y_max=0.0), dict(y_max=0.05, w=0.01, theta=-0.02), dict(theta=-1e6, lam=0.5, y_max=0.0), dict(lam=0.5),
], ids=lambda d: ",".join(f"{k}={v}" for k, v in d.items()))
def test_parameter_strain(O, variant, kw):
    code = wl.peg_code(504, 252, 3, seed=3)
    y, _, sig = wl.frames(code, 40, 2.5, seed=8)
    base = dict(lam=0.97, t_max=30, smooth_window=10)
    base.update(kw)
    for prec in PREC:
        if prec.get("q_bits") and not base.get("y_max", 2.5) > 0:
            continue                                    # fixed point needs a finite saturation
        if prec.get("precision") == ngdbf.NGDBF_FIXACC and abs(base.get("theta", 0.9)) > 1e5:
            continue                                    # beyond the accumulator's range
        assert_parity(O, code, y, sig, seed=6, variant=variant, **base, **prec)


@pytest.mark.parametrize("variant", [0, 3, 4])
def test_non_finite_and_large_samples(O, variant):
    code = wl.peg_code(504, 252, 3, seed=3)
    y, _, sig = wl.frames(code, 40, 3.0, seed=9)
    rng = np.random.default_rng(4)
    at = rng.random(y.shape)
    y[at < 0.01] = np.inf
    y[(at >= 0.01) & (at < 0.02)] = -np.inf
    y[(at >= 0.02) & (at < 0.03)] *= 1e30
    y[(at >= 0.03) & (at < 0.04)] = 0.0
    for y_max in (2.5, 0.0):
        assert_parity(O, code, y, sig, seed=6, variant=variant, lam=0.97, t_max=30, smooth_window=10, y_max=y_max)
    assert_parity(O, code, y, sig, seed=6, variant=variant, lam=0.97, t_max=30, smooth_window=10,
                  precision=ngdbf.NGDBF_FP16)


@pytest.mark.parametrize("F", [1, 2, 3, 5, 9, 16, 17, 31])
@pytest.mark.parametrize("variant", [0, 3, 6])
def test_live_slots(O, F, variant):
    """Few live slots in a CTA: lanes cover several groups of the same slot."""
    code = wl.code_from_dense(wl.peg_code(512, 256, 3, seed=2).dense()[:, :509])
    y, _, sig = wl.frames(code, F, 2.5, seed=F)
    assert_parity(O, code, y, sig, seed=1, frame_offset=2 ** 32 - 7, variant=variant, lam=0.97, t_max=60, smooth_window=10)


@pytest.mark.parametrize("variant", [0, 3, 4])
def test_longest_codes(O, variant):
    """A code whose arrays fit shared memory only with the queues over the syndrome words."""
    n, m = 10950, 300
    H = np.zeros((m, n), np.uint8)
    H[np.arange(n) % m, np.arange(n)] = 1
    code = wl.code_from_dense(H)
    y, _, _ = wl.frames(code, 40, None, seed=5, sigma=0.8)
    assert_parity(O, code, y, 0.8, seed=2, variant=variant, lam=0.95, t_max=8, smooth_window=3, w=0.4, theta=-0.5)
