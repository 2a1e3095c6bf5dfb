"""Many live slots per CTA vs the reference decoder, bit for bit.

A batch is spread over the CTAs that can be resident, so that a CTA holds more than one frame only
when there are more frames than CTAs.  Frame counts here are multiples of the launch's largest
grid, which gives every CTA the slots under test from its first iteration on: lanes over (group,
slot) below 32 of them, the warps' queues and pairs of groups from 17 on, and flips of several
slots in one iteration on both sides of the number up to which they are recorded.
"""
import numpy as np
import pytest

from paper_1402_2773_gb300 import ngdbf, workload as wl
from test_gpu_parity import O, _gpu, gpu_decode, irregular_code, params_pair, THREADS  # noqa: F401
from test_z_lazy import PREC

pytestmark = pytest.mark.gpu


def assert_slots(O, code, slots, sigma, seed=1, rest=0, amplitude=1.0, **kw):
    """Parity of a batch that gives every CTA `slots` frames at first (`rest` more frames follow)."""
    gp, op = params_pair(**kw)
    gpu_decode(code, np.ones((20000, code.n), np.float32), sigma, gp, seed)     # all checks satisfied: t = 0 only
    grid = ngdbf.ngdbf_last_launch()["grid"]
    assert grid < 20000
    F = grid * slots + rest
    rng = np.random.default_rng(seed + 100)
    y = (amplitude + sigma * rng.standard_normal((F, code.n))).astype(np.float32)
    g = gpu_decode(code, y, sigma, gp, seed)
    launch = ngdbf.ngdbf_last_launch()
    assert launch["grid"] == grid and -(-F // grid) == slots + (1 if rest else 0)
    o = O.decode_f32(code, y, sigma, op, seed=seed, threads=THREADS)
    bad = np.nonzero((g[0] != o[0]).any(axis=1) | (g[1] != o[1]) | (g[2] != o[2]))[0]
    assert bad.size == 0, f"{bad.size}/{F} frames differ, first {bad[:5]}"
    return o


FLIPS = wl.peg_code(504, 252, 3, seed=3)


@pytest.mark.parametrize("theta", [-1.5, -1.2, -0.9, -0.6])
@pytest.mark.parametrize("variant", [0, 3])
def test_flips_about_the_recorded_number(O, theta, variant):
    """32 slots, from a few flips an iteration of a CTA to some hundred: the count passes the limit
    up to which flips are recorded while warps still add theirs."""
    assert_slots(O, FLIPS, 32, 0.55, variant=variant, lam=0.99, t_max=12, smooth_window=4, w=0.5, theta=theta, eta=0.9)


SMALL = irregular_code(203, 101, seed=5)
BASE = dict(lam=0.97, t_max=10, smooth_window=4, w=0.5, theta=-0.7, eta=0.9)


@pytest.mark.parametrize("slots", [2, 5, 17, 31, 32])
@pytest.mark.parametrize("k,variant", list(enumerate([0, 3, 4, 6, 3 | 8])))
def test_live_slots_per_cta(O, slots, k, variant):
    """Some more frames than slots, so that slots are refilled at different iterations."""
    prec = PREC[(k + slots) % 4]
    assert_slots(O, SMALL, slots, 0.6, rest=77, variant=variant, **BASE, **prec)


@pytest.mark.parametrize("variant", [0, 3, 4])
@pytest.mark.parametrize("kw", [dict(w=1e-3), dict(w=20.0), dict(theta=0.4), dict(eta=0.0), dict(y_max=0.05, w=0.01, theta=-0.02),
                                dict(theta=-1e6, lam=0.5, y_max=0.0)], ids=lambda d: ",".join(f"{k}={v}" for k, v in d.items()))
def test_strain_with_full_slots(O, kw, variant):
    d = dict(BASE)
    d.update(kw)
    assert_slots(O, SMALL, 32, 0.6, variant=variant, **d)
