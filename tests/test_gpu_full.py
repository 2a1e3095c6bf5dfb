"""Batches so noisy that most outputs are at or below their cutoffs, vs the reference decoder, bit for
bit: in the adaptive variants CTAs with more than half of their slots live go over from the lazy
form to one that forms every E_k and back, with frames that finish, are refilled or run out on both sides of it.
"""
import numpy as np
import pytest

from paper_1402_2773_gb300 import ngdbf, workload as wl
from test_gpu_limits import serve
from test_gpu_parity import O, _gpu, gpu_decode, irregular_code, params_pair, THREADS  # noqa: F401
from test_z_lazy import PREC

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

IDS = ["fp32", "fp16", "fix3", "fixacc8"]
# a length that is a multiple of neither 4 nor 8 (a single last group of one symbol, degrees to 5), and
# one whose last pair of groups is whole
RAGGED, EVEN = irregular_code(205, 101, seed=5), wl.peg_code(504, 252, 3, seed=3)
KW = dict(lam=0.99, smooth_window=12, w=0.75, theta=-0.9, eta=0.95)


def noisy(code, F, seed, clean=0.25):
    """Samples of pure noise, and for a share of the frames ones that are decoded in a few iterations."""
    rng = np.random.default_rng(seed)
    s = np.where(rng.random(F) < clean, 0.5, 2.5)[:, None]
    return (np.where(s < 1, 1.0, 0.0) + s * rng.standard_normal((F, code.n))).astype(np.float32)


def grid_of(code, gp):
    gpu_decode(code, np.ones((20000, code.n), np.float32), 0.8, gp, 1)
    return ngdbf.ngdbf_last_launch()["grid"]


@pytest.mark.parametrize("prec", PREC, ids=IDS)
@pytest.mark.parametrize("variant", [0, 1, 2, 3, 3 | 8])
@pytest.mark.parametrize("code,per", [(RAGGED, 32), (EVEN, 24)], ids=["ragged", "even"])
def test_noise(O, code, per, variant, prec):
    gp, op = params_pair(variant=variant, t_max=45, **KW, **prec)
    F = grid_of(code, gp) * per + 333
    y = noisy(code, F, seed=variant)
    got = gpu_decode(code, y, 0.8, gp, 7, 2 ** 32 - 1000)
    want = O.decode_f32(code, y, 0.8, op, seed=7, frame_offset=2 ** 32 - 1000, threads=THREADS)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("variant", [0, 3])
def test_state_in_global_memory(O, variant):
    code = wl.peg_code(4096, 2048, 4, seed=1)
    gp, op = params_pair(variant=variant, t_max=22, **KW)
    y = noisy(code, 152 * 20, seed=3)
    got = gpu_decode(code, y, 0.8, gp, 7)
    for a, b in zip(got, O.decode_f32(code, y, 0.8, op, seed=7, threads=THREADS)):
        assert np.array_equal(a, b)


def test_longest_code(O):
    n, m = 10900, 300
    H = np.zeros((m, n), np.uint8)
    H[np.arange(n) % m, np.arange(n)] = 1
    code = wl.code_from_dense(H)
    gp, op = params_pair(variant=3, t_max=20, **KW)
    y = noisy(code, 152 * 18, seed=4, clean=0.0)
    got = gpu_decode(code, y, 0.8, gp, 7)
    for a, b in zip(got, O.decode_f32(code, y, 0.8, op, seed=7, threads=THREADS)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", PREC, ids=IDS)
def test_table(O, prec):
    made, codes = [], []
    for j, (code, F) in enumerate([(RAGGED, 9000), (EVEN, 9001)]):
        gp, op = params_pair(variant=3, t_max=40, **KW, **prec)
        y = noisy(code, F, seed=20 + j)
        codes.append(ngdbf.DeviceCode.from_code(code))
        made.append((codes[-1], y, gp, 1000 * j, O.decode_f32(code, y, 0.8, op, seed=9, frame_offset=1000 * j, threads=THREADS)))
    batch = ngdbf.Batch([(dc, torch.from_numpy(y).cuda(), 0.8, gp, off) for dc, y, gp, off, _ in made], seed=9)
    try:
        for k, _ in enumerate(batch.shapes()):
            batch.use_shape(k)
            got = batch.launch()
            torch.cuda.synchronize()
            for g, q in zip(got, made):
                for a, b in zip(g, q[4]):
                    assert np.array_equal(a.cpu().numpy(), b)
                    a.zero_()
    finally:
        batch.close()
        for dc in codes:
            dc.close()


@pytest.mark.parametrize("variant", [0, 3])
def test_server(O, variant):
    """Requests of two codes, most too small for a CTA's slots: frames of several share them."""
    reqs, want = [], []
    for j in range(60):
        code, F = (RAGGED, 40) if j % 2 else (EVEN, 12 + j)
        gp, op = params_pair(variant=variant, t_max=40, **KW)
        y, sigma = noisy(code, F, seed=40 + j), 0.8 + 0.002 * j
        reqs.append((code, y, sigma, gp, 1000 * j))
        want.append(O.decode_f32(code, y, sigma, op, seed=9, frame_offset=1000 * j, threads=THREADS))
    outs, status = serve(reqs, seed=9)
    assert status == [0] * len(reqs)
    for got, ref in zip(outs, want):
        for a, b in zip(got, ref):
            assert np.array_equal(a, b)
