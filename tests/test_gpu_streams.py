"""Small decodes on several streams at once: a launch that finds others' frames on the device packs its
own more densely, and the results are those of the same calls one after another.
"""
import numpy as np
import pytest

from paper_1402_2773_gb300 import ngdbf, workload as wl
from test_gpu_parity import O, _gpu, params_pair, THREADS  # noqa: F401
from test_z_lazy import code_with_degree

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [0, 3, 4])
def test_many_streams(O, variant):
    codes = [wl.peg_code(504, 252, 3, seed=3), wl.code_c2(), code_with_degree(150, 80, 20, seed=20)]
    handles = [ngdbf.DeviceCode.from_code(c) for c in codes]
    calls = []
    gp, op = params_pair(variant=variant, lam=0.99, t_max=60, smooth_window=12, w=0.3, theta=-0.7, eta=0.8)
    for j, F in enumerate([1, 7, 33, 96, 150, 40, 96, 64, 5, 200, 96, 31] * 2):
        c = j % 3
        y, _, sig = wl.frames(codes[c], F, None, seed=j, sigma=0.6)
        calls.append((c, torch.from_numpy(y).cuda(), F, O.decode_f32(codes[c], y, 0.6, op, seed=5, frame_offset=j, threads=THREADS)))
    streams = [torch.cuda.Stream() for _ in range(12)]
    torch.cuda.synchronize()
    try:
        for _ in range(3):
            outs = []
            for j, (c, y, F, _) in enumerate(calls):
                with torch.cuda.stream(streams[j % 12]):
                    outs.append(handles[c].decode(y, 0.6, gp, seed=5, frame_offset=j))
            torch.cuda.synchronize()
            for (c, y, F, want), got in zip(calls, outs):
                for a, b in zip(got, want):
                    assert np.array_equal(a.cpu().numpy(), b)
    finally:
        for h in handles:
            h.close()
