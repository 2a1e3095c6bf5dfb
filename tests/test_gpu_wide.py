"""Symbol degrees above 15 (bit-sliced counts, every E_k formed) through every kernel vs the
reference decoder, bit for bit: single launches with full slots, job tables that hold narrow and
wide codes in every launch shape (clusters too), and the server.  A small batch of such a code
is packed 32 frames to a CTA, whose time does not depend on its live slots.
"""
import numpy as np
import pytest

from paper_1402_2773_gb300 import ngdbf, workload as wl
from test_gpu_limits import serve
from test_gpu_parity import O, _gpu, gpu_decode, params_pair, THREADS  # noqa: F401
from test_gpu_slots import assert_slots
from test_z_lazy import PREC, code_with_degree

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

W16, W20, W64 = (code_with_degree(150, 80, t, seed=t) for t in (16, 20, 64))
LONG16 = code_with_degree(2100, 700, 16, seed=3)
NARROW, LONG3 = wl.peg_code(504, 252, 3, seed=3), wl.peg_code(2200, 1100, 3, seed=4)
KW = dict(lam=0.97, t_max=12, smooth_window=5, w=0.3, theta=-0.6)


def job(O, code, F, variant, prec, j):
    gp, op = params_pair(variant=variant, **KW, **prec)
    y, _, _ = wl.frames(code, F, None, seed=70 + j, sigma=0.6)
    return (code, y, gp, 1000 * j, O.decode_f32(code, y, 0.6, op, seed=9, frame_offset=1000 * j, threads=THREADS))


@pytest.mark.parametrize("F", [1, 32, 33, 96, 500])
def test_small_batches_are_packed(O, F):
    gp, op = params_pair(variant=3, **KW)
    y, _, _ = wl.frames(W20, F, None, seed=7, sigma=0.6)
    got = gpu_decode(W20, y, 0.6, gp, 3)
    assert ngdbf.ngdbf_last_launch()["grid"] == (F + 31) // 32
    for a, b in zip(got, O.decode_f32(W20, y, 0.6, op, seed=3, threads=THREADS)):
        assert np.array_equal(a, b)


def test_small_jobs_of_a_table_are_packed(O):
    """The first shape (no cluster): a CTA per 32 frames of each job."""
    made = [job(O, code, F, 3, {}, j) for j, (code, F) in enumerate([(W20, 33), (W16, 64), (NARROW, 70)])]
    codes = [ngdbf.DeviceCode.from_code(q[0]) for q in made]
    batch = ngdbf.Batch([(dc, torch.from_numpy(q[1]).cuda(), 0.6, q[2], q[3]) for dc, q in zip(codes, made)], seed=9)
    try:
        batch.use_shape(0)
        got = batch.launch()
        torch.cuda.synchronize()
        assert ngdbf.ngdbf_last_launch()["grid"] == 2 + 2 + 3
        for g, q in zip(got, made):
            for a, b in zip(g, q[4]):
                assert np.array_equal(a.cpu().numpy(), b)
    finally:
        batch.close()
        for dc in codes:
            dc.close()


@pytest.mark.parametrize("prec", PREC, ids=["fp32", "fp16", "fix3", "fixacc8"])
@pytest.mark.parametrize("variant", [0, 3, 6])
def test_full_slots(O, variant, prec):
    for code in (W16, W64):
        assert_slots(O, code, 32, 0.6, rest=41, variant=variant, **KW, **prec)


@pytest.mark.parametrize("prec", PREC[:2], ids=["fp32", "fp16"])
@pytest.mark.parametrize("variant", [0, 3, 6])
def test_tables_of_narrow_and_wide_codes(O, variant, prec):
    """In a table with one wide code every job is decoded in the wide format; the jobs of 2048 symbols
    and more are split over clusters in some shapes."""
    made = [job(O, code, F, variant, prec, j) for j, (code, F) in enumerate([(NARROW, 70), (W20, 33), (LONG16, 40), (LONG3, 65)])]
    codes = [ngdbf.DeviceCode.from_code(q[0]) for q in made]
    batch = ngdbf.Batch([(dc, torch.from_numpy(q[1]).cuda(), 0.6, q[2], q[3]) for dc, q in zip(codes, made)], seed=9)
    try:
        clusters = set()
        for k, shape in enumerate(batch.shapes()):
            batch.use_shape(k)
            clusters.add(shape["cluster"])
            got = batch.launch()
            torch.cuda.synchronize()
            for g, q in zip(got, made):
                for a, b in zip(g, q[4]):
                    assert np.array_equal(a.cpu().numpy(), b), shape
                    a.zero_()
        assert len(clusters) > 1
    finally:
        batch.close()
        for dc in codes:
            dc.close()


@pytest.mark.parametrize("prec", PREC, ids=["fp32", "fp16", "fix3", "fixacc8"])
def test_server_of_narrow_and_wide_codes(O, prec):
    for variant in (3, 4):
        made = [job(O, code, F, variant, prec, j) for j, (code, F) in enumerate(
            [(W20, 3), (NARROW, 40), (LONG16, 35), (W16, 50), (LONG3, 5), (W64, 33), (W20, 64), (LONG16, 2)] + [(W16, 3)] * 18)]
        outs, status = serve([(q[0], q[1], 0.6, q[2], q[3]) for q in made], seed=9)
        assert status == [0] * len(made)
        for got, q in zip(outs, made):
            for a, b in zip(got, q[4]):
                assert np.array_equal(a, b)
