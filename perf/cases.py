"""The decode calls whose time matters to a user of this library, with their inputs.

Codes, parameter sets, frame counts and Eb/N0 points are those of the benchmark (bench.py), the
precision study and the tests; every case goes through the public binding in
paper_1402_2773_gb300.ngdbf.  Inputs are random codewords (encoded on the GPU with the code's
systematic encoder), BPSK, AWGN of the stated Eb/N0, FP32 samples.
"""
import atexit
import functools
import math

import numpy as np
import torch

from paper_1402_2773_gb300 import ngdbf
from paper_1402_2773_gb300 import workload as wl

# (n, m, d_v) of the seeded PEG codes, the rate-1/2 and high-rate shapes of the paper's experiments
PEG = {"n504": (504, 252, 3), "n1008": (1008, 504, 3), "n4096": (4096, 2048, 4), "n2048": (2048, 384, 6),
       "n8192": (8192, 1639, 3)}
TABLE_CODES = "n504,n1008,n4096,n2048,n8192"
HIGH_RATE = dict(w=0.1875, theta=-0.7, eta=0.65, lam=0.993, y_max=2.0)      # Fig. 5 set, the (6,32) code
RATE_HALF = dict(w=0.75, theta=-0.9, eta=0.95, lam=0.99, y_max=2.5)         # Figs. 2-4 set
LARGE_DV3 = dict(w=0.5, theta=-0.7, eta=0.8, lam=0.99, y_max=2.5)           # the (3,15) code
PRECISION = {"fp32": (ngdbf.NGDBF_FP32, 0), "fp16": (ngdbf.NGDBF_FP16, 0), "fix8": (ngdbf.NGDBF_FIXACC, 8),
             "fix8-eq9": (ngdbf.NGDBF_FIX, 8)}
SM, PLAIN, ADAPT, SMOOTH, SINGLE = 3, 0, 1, 2, 4


def _case(name, entry, code, frames, ebn0, t_max, window=64, variant=SM, precision="fp32"):
    return dict(name=name, entry=entry, code=code, frames=frames, ebn0=ebn0, t_max=t_max, window=window,
                variant=variant, precision=precision)


def listed():
    return [
        # one received word of the (3,6) N=1008 code: the least a receiver asks for, all latency
        _case("one frame", "device", "n1008", 1, 3.5, 80, 32),
        # a short burst of the high-rate code: three 32-frame groups, far fewer than the GPU holds
        _case("burst of 96", "device", "n2048", 96, 4.0, 300),
        # the plain non-adaptive decoder of the precision study (no per-symbol state)
        _case("plain rate 1/2", "device", "n1008", 20000, 4.0, 100, 64, PLAIN),
        # the single-bit decoder (S-NGDBF, one flip per iteration)
        _case("single-bit", "device", "n1008", 4096, 4.5, 100, 20, SINGLE),
        # the benchmark's decoder at its hardest point, most frames running to T: the largest batch
        _case("bench 3.5 dB", "device", "n2048", 200000, 3.5, 300),
        # the same decoder in binary16 at the middle point
        _case("fp16 4.0 dB", "device", "n2048", 60000, 4.0, 300, 64, SM, "fp16"),
        # 8-bit held samples at the easiest point, an odd frame count
        _case("fix8 4.5 dB", "device", "n2048", 100003, 4.5, 300, 64, SM, "fix8"),
        # a long code whose state does not fit shared memory
        _case("long code", "device", "n8192", 1073, 3.7, 171),
        # an irregular code of odd length with a symbol of degree 9 (the wide count format)
        _case("odd irregular", "device", "irregular203", 3001, 3.0, 40, 9),
        # host buffers in and out: copies in, decode, copies back
        _case("host buffers", "host", "n2048", 32768, 4.0, 300),
        # five codes in one job-table launch (bench.py --workload multicode)
        _case("five-code table", "table", TABLE_CODES, 1024, 4.0, 200),
        # a burst of requests of five codes to a running server, host buffers
        _case("server burst", "server", TABLE_CODES, 512, 4.0, 200),
    ]


def draw(rng):
    entry = rng.choice(["device"] * 7 + ["host", "table", "server"])
    lo, hi = 3.0, 5.0
    if entry in ("table", "server"):
        names = rng.sample(sorted(PEG), rng.randint(2, 5))
        return dict(entry=entry, code=",".join(names), frames=int(round(math.exp(rng.uniform(math.log(16), math.log(2000))))),
                    ebn0=round(rng.uniform(3.5, 4.5), 3), t_max=rng.randint(100, 300), window=64, variant=SM, precision="fp32")
    code = rng.choice(["n504", "n1008", "n1008", "n2048", "n2048", "n4096", "n8192", "irregular203", "peg2598"])
    variant = rng.choice([SM, SM, SM, PLAIN, ADAPT, SMOOTH, SINGLE, SM | ngdbf.NGDBF_UNIFORM])
    t_max = rng.randint(40, 300) if variant & SM else rng.randint(40, 120)
    n = {"irregular203": 203, "peg2598": 2598}.get(code) or PEG[code][0]
    most = min(200000, int(2.5e10 / (n * t_max)))           # costs at most about half of the largest listed case
    least = 1 if entry == "device" else 1000
    frames = int(round(math.exp(rng.uniform(math.log(least), math.log(max(most, least + 1))))))
    return dict(entry=entry, code=code, frames=frames, ebn0=round(rng.uniform(lo, hi), 3), t_max=t_max,
                window=rng.randint(0, 64), variant=variant,
                precision=rng.choice(["fp32", "fp32", "fp32", "fp16", "fix8", "fix8-eq9"]))


# --- inputs ----------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _code(name):
    if name in PEG:
        n, m, dv = PEG[name]
        return wl.peg_code(n, m, dv, seed=1)
    if name == "peg2598":           # a length that is a multiple of neither 4 nor 32
        H = wl.peg_code(2600, 1300, 3, seed=2).dense()[:, :2598]
        return wl.code_from_dense(np.ascontiguousarray(H))
    n, m = 203, 101                 # irregular203: symbol degrees 2..5 and one of 9
    rng = np.random.default_rng(5)
    H = np.zeros((m, n), np.uint8)
    for k in range(n):
        H[rng.choice(m, size=int(rng.integers(2, 6)), replace=False), k] = 1
    H[:9, 0] = 1
    for i in np.nonzero(H.sum(1) == 0)[0]:
        H[i, rng.integers(n)] = 1
    return wl.code_from_dense(H)


@functools.lru_cache(maxsize=None)
def _device_code(name):
    return ngdbf.DeviceCode.from_code(_code(name))


@functools.lru_cache(maxsize=None)
def _encoder(name):
    """Information and pivot positions and the parity matrix [K, rank], on the GPU."""
    e = _code(name).encoder()
    P = np.unpackbits(e.pmask.view(np.uint8), axis=1, bitorder="little")[:, :e.k]
    dev = "cuda"
    return (torch.from_numpy(e.info_pos.astype(np.int64)).to(dev), torch.from_numpy(e.pivot_pos.astype(np.int64)).to(dev),
            torch.from_numpy(np.ascontiguousarray(P.T).astype(np.float32)).to(dev))


def _sigma(name, ebn0):
    return wl.sigma_for(ebn0, _code(name).rate)


def _samples(name, frames, ebn0, seed):
    """float32 CUDA tensor [frames, n]: random codewords through the AWGN channel."""
    info, pivot, P = _encoder(name)
    n, sigma = _code(name).n, _sigma(name, ebn0)
    g = torch.Generator(device="cuda").manual_seed(seed)
    y = torch.empty((frames, n), dtype=torch.float32, device="cuda")
    for s in range(0, frames, 16384):
        F = min(16384, frames - s)
        u = torch.randint(0, 2, (F, info.numel()), generator=g, device="cuda").float()
        c = torch.empty((F, n), dtype=torch.float32, device="cuda")
        c[:, info] = u
        c[:, pivot] = torch.remainder(u @ P, 2.0)           # sums of at most 2^13 ones: exact
        part = y[s:s + F]
        part.normal_(generator=g)
        part.mul_(sigma).add_(1.0 - 2.0 * c)
    return y


def _params(name, case):
    prec, q_bits = PRECISION[case["precision"]]
    code = _code(name)
    base = HIGH_RATE if name == "n2048" else LARGE_DV3 if code.rate > 0.7 else RATE_HALF
    kw = dict(base)
    if case["variant"] & SINGLE:
        kw.update(eta=1.0)
    elif name == "n4096":
        kw.update(eta=0.7)
    elif not case["variant"] & ADAPT:
        kw.update(eta=0.96 if base is RATE_HALF else kw["eta"])
    return ngdbf.make_params(**kw, t_max=case["t_max"], smooth_window=case["window"], variant=case["variant"],
                             precision=prec, q_bits=q_bits)


def _outputs(name, frames, **where):
    n = _code(name).n
    return (torch.empty((frames, (n + 7) // 8), dtype=torch.uint8, **where),
            torch.empty(frames, dtype=torch.int32, **where), torch.empty(frames, dtype=torch.uint8, **where))


def _host(t):
    """A page-locked host copy from the library's allocator."""
    h = ngdbf.host_empty(tuple(t.shape), np.float32)
    h.copy_(t)
    return h


def _parts(case):
    """(code, frames, Eb/N0) of each job or request: uneven counts around case["frames"], fixed by the case."""
    names = case["code"].split(",")
    rng = np.random.default_rng(case["frames"])
    per = 1 if case["entry"] == "table" else 4
    return [(name, int(np.clip(rng.exponential(case["frames"]), 1, 4 * case["frames"])),
             case["ebn0"] + float(rng.uniform(-0.5, 0.5))) for _ in range(per) for name in names]


@functools.lru_cache(maxsize=None)
def _server():
    """The server a program keeps running (its perturbation seed is its own)."""
    srv = ngdbf.Server(8 << 30, max_inflight=4, max_jobs=256, seed=1)
    atexit.register(srv.close)
    return srv


def prepare(case, seed):
    seed = int(seed)
    if case["entry"] == "table":
        jobs = [(_device_code(name), _samples(name, F, eb, seed * 64 + j), _sigma(name, eb), _params(name, case), 10 ** 7 * j)
                for j, (name, F, eb) in enumerate(_parts(case))]
        return dict(entry="table", batch=ngdbf.Batch(jobs, seed=seed, flags=ngdbf.NGDBF_BATCH_GRAPH | ngdbf.NGDBF_BATCH_TUNE))
    if case["entry"] == "server":
        reqs = [dict(code=_device_code(name), y=_host(_samples(name, F, eb, seed * 64 + j)), sigma=_sigma(name, eb),
                     params=_params(name, case), offset=10 ** 9 * (j + 1), out=_outputs(name, F, pin_memory=True))
                for j, (name, F, eb) in enumerate(_parts(case))]
        return dict(entry="server", server=_server(), requests=reqs)
    name, F = case["code"], case["frames"]
    y = _samples(name, F, case["ebn0"], seed)
    state = dict(entry=case["entry"], code=_device_code(name), sigma=_sigma(name, case["ebn0"]), params=_params(name, case),
                 seed=seed)
    if case["entry"] == "host":
        return dict(state, y=_host(y), out=_outputs(name, F, pin_memory=True))
    return dict(state, y=y, out=_outputs(name, F, device="cuda"))


def run(state):
    if state["entry"] == "table":
        return state["batch"].launch()
    if state["entry"] == "server":
        srv = state["server"]
        for r in state["requests"]:
            srv.submit(r["code"], r["y"], r["sigma"], r["params"], frame_offset=r["offset"], out=r["out"])
        srv.wait(600)
        srv.poll()
        return [r["out"] for r in state["requests"]]
    decode = state["code"].decode_host if state["entry"] == "host" else state["code"].decode
    return decode(state["y"], state["sigma"], state["params"], seed=state["seed"], out=state["out"])


def work(case):
    """Samples read and outputs written once; the operations of one iteration of every frame (how
    many more a frame needs depends on its noise): generator, inversion function, comparison and
    counters, and the d_v checks of every symbol."""
    parts = _parts(case) if case["entry"] in ("table", "server") else [(case["code"], case["frames"], case["ebn0"])]
    by = fl = 0
    for name, F, _ in parts:
        c = _code(name)
        by += F * (4 * c.n + (c.n + 7) // 8 + 5)
        fl += F * (46 * c.n + 2 * int(c.row_ptr[-1]))
    return {"bytes": float(by), "flops": float(fl)}


def exact(case, seed):
    """Every output is a decision, an iteration count or a pass flag: none is a computed real number."""
    return None
