"""The longest codes through every entry point that takes device memory plans of its own, vs the
reference decoder, bit for bit: a job table and the server.
"""
import numpy as np
import pytest

from paper_1402_2773_gb300 import ngdbf, workload as wl
from test_gpu_parity import O, _gpu, params_pair, THREADS  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def long_code(n, m):
    """Symbols of degree 1 (check degrees up to 64)."""
    H = np.zeros((m, n), np.uint8)
    H[np.arange(n) % m, np.arange(n)] = 1
    return wl.code_from_dense(H)


LONGEST = [(11000, 172), (10900, 300), (10160, 1000)]


def serve(reqs, seed):
    """The outputs and statuses of requests (code, y, sigma, params, offset) to a new server."""
    srv = ngdbf.Server(4 << 30, max_inflight=2, max_jobs=64, seed=seed)
    codes, outs = {}, []
    try:
        for code, y, sigma, gp, off in reqs:
            dc = codes.setdefault(id(code), None) or ngdbf.DeviceCode.from_code(code)
            codes[id(code)] = dc
            F = y.shape[0]
            out = (np.empty((F, (code.n + 7) // 8), np.uint8), np.empty(F, np.int32), np.empty(F, np.uint8))
            outs.append(out)
            srv.submit(dc, y, sigma, gp, frame_offset=off, out=out)
        srv.wait(120)
        return outs, [r[2] for r in srv.poll()]
    finally:
        srv.close()
        for c in codes.values():
            c.close()


@pytest.mark.parametrize("n,m", LONGEST)
def test_server_takes_the_longest_codes(O, n, m):
    code = long_code(n, m)
    reqs, want = [], []
    for j in range(20):                                 # enough for requests to share a CTA's slots
        gp, op = params_pair(variant=3, lam=0.95, t_max=6, smooth_window=3, w=0.4, theta=-0.5)
        y, _, _ = wl.frames(code, 3, None, seed=30 + j, sigma=0.7 + 0.01 * j)
        reqs.append((code, y, 0.7 + 0.01 * j, gp, 1000 * j))
        want.append(O.decode_f32(code, y, 0.7 + 0.01 * j, op, seed=4, frame_offset=1000 * j, threads=THREADS))
    outs, status = serve(reqs, seed=4)
    assert status == [0] * len(reqs)
    for got, ref in zip(outs, want):
        for a, b in zip(got, ref):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("n,m", LONGEST)
def test_table_takes_the_longest_codes(O, n, m):
    jobs, want, codes = [], [], []
    for j, code in enumerate([long_code(n, m), wl.peg_code(504, 252, 3, seed=3)]):
        gp, op = params_pair(variant=3, lam=0.95, t_max=6, smooth_window=3, w=0.4, theta=-0.5)
        y, _, _ = wl.frames(code, 70, None, seed=30 + j, sigma=0.7)
        codes.append(ngdbf.DeviceCode.from_code(code))
        jobs.append((codes[-1], torch.from_numpy(y).cuda(), 0.7, gp, 1000 * j))
        want.append(O.decode_f32(code, y, 0.7, op, seed=4, frame_offset=1000 * j, threads=THREADS))
    batch = ngdbf.Batch(jobs, seed=4)
    try:
        got = batch.launch()
        torch.cuda.synchronize()
        for g, ref in zip(got, want):
            for a, b in zip(g, ref):
                assert np.array_equal(a.cpu().numpy(), b)
    finally:
        batch.close()
        for c in codes:
            c.close()


def test_codes_whose_maxima_do_not_fit_together(O):
    """Two codes that fit alone, one of many symbols and one of many checks: a kernel for both would
    need more shared memory than there is, so the server serves them in turn."""
    A = long_code(9300, 930)
    H = np.zeros((5590, 5600), np.uint8)
    H[np.arange(5600) % 5590, np.arange(5600)] = 1
    H[10:20, 0] = 1
    B = wl.code_from_dense(H)
    reqs, want = [], []
    for j, code in enumerate([A, B, A, B, B, A]):
        gp, op = params_pair(variant=3, lam=0.95, t_max=6, smooth_window=3, w=0.4, theta=-0.5)
        y, _, _ = wl.frames(code, 4, None, seed=50 + j, sigma=0.7)
        reqs.append((code, y, 0.7, gp, 100 * j))
        want.append(O.decode_f32(code, y, 0.7, op, seed=4, frame_offset=100 * j, threads=THREADS))
    outs, status = serve(reqs, seed=4)
    assert status == [0] * len(reqs)
    for got, ref in zip(outs, want):
        for a, b in zip(got, ref):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("n,m,block", [(11000, 172, 256), (10950, 300, 512), (10600, 700, 1024)])
def test_threads_of_the_longest_codes(O, n, m, block):
    """As many warps as there are syndrome words for their queues."""
    code = long_code(n, m)
    gp, op = params_pair(variant=3, lam=0.95, t_max=8, smooth_window=3, w=0.4, theta=-0.5)
    y, _, _ = wl.frames(code, 152 * 3, None, seed=5, sigma=0.8)
    dc = ngdbf.DeviceCode.from_code(code)
    try:
        got = dc.decode(torch.from_numpy(y).cuda(), 0.8, gp, seed=2)
        torch.cuda.synchronize()
        assert ngdbf.ngdbf_last_launch()["block"] == block
    finally:
        dc.close()
    for a, b in zip(got, O.decode_f32(code, y, 0.8, op, seed=2, threads=THREADS)):
        assert np.array_equal(a.cpu().numpy(), b)
