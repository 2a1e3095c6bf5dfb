"""Shared-memory layouts of the lazy evaluation (host side, no GPU).

Every array of a layout is placed, aligned, in order and inside its total, and none overlaps
another but the warps' queues over the syndrome words of the longest codes; the counts can be read
31 groups past the code's.  And no code that fitted before the lazy arrays were added is refused:
the former layouts (without them, 16 bytes of syndromes per check and 4-bit counts up to degree 7)
are stated here, with the former static shared memory of each kernel.
"""
import os
import shutil
import subprocess

import pytest

from paper_1402_2773_gb300 import _build

SRC = r"""
#include "ngdbf_kernels.cuh"
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <algorithm>
#include <cstdint>

using namespace ngdbf;

static uint64_t s = 0;
static uint32_t rnd() {            // splitmix64
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return (uint32_t)((z ^ (z >> 31)) >> 32);
}
static int in(int lo, int hi) { return lo + (int)(rnd() % (uint32_t)(hi - lo + 1)); }

struct Span { const char* name; int at, bytes; };

// Every array of L with the bytes the kernel uses of it.
static bool sane(const SmemLayout& L, int n, int m, int nl, int dv, int dc, bool thr, bool st, int tables, bool wide,
                 int use, int warps) {
    const bool serve = use > kTable, tight = tables & kTight;
    Span a[] = {{"frame", L.off_frame, kSlots * 8}, {"start", L.off_start, kSlots * 4}, {"ctl", L.off_ctl, 32},
                {"unsat", wide ? -1 : L.off_unsat, kSlots * 4}, {"best", L.off_best, (serve ? 1 : 2) * kSlots * 8},
                {"tau", wide ? -1 : L.off_tau, kSlots * 4}, {"trace", use == kLaunch ? L.off_trace : -1, kSlots * 12},
                {"icdf", L.off_icdf, 4096}, {"cut", wide ? -1 : L.off_cut, L.cuts * 1024},
                {"cnt", L.off_cnt, pad4(nl) * (wide ? 32 : 16)}, {"flips", wide || tight ? -1 : L.off_flips, kFlips * 4},
                {"queue", wide || tight ? -1 : L.off_queue, 32 * kQueue * 4}, {"xw", L.off_xw, pad4(n + 1) * 4},
                {"sw", L.off_sw, (m + 1) * (wide ? 4 : 8)}, {"thr", thr ? L.off_thr : -1, 2048},
                {"st", st ? L.off_st : -1, pad4(nl) * kSlots * 2},
                {"chk", tables & kTabChk ? L.off_chk : -1, chk_entries(m, dc) * 2},
                {"sym", tables & kTabSym ? L.off_sym : -1, pad4(nl) * dv * 2 + nl}};
    const char* must[] = {"frame", "start", "ctl", "best", "icdf", "cnt", "xw", "sw"};
    for (const Span& x : a) {
        for (const char* q : must)
            if (!strcmp(q, x.name) && x.at < 0) { printf("FAIL %s not placed\n", q); return false; }
        if (x.at < 0) continue;
        if (x.at % 16 || x.at + x.bytes > L.total) { printf("FAIL %s: %d + %d of %d\n", x.name, x.at, x.bytes, L.total); return false; }
        for (const Span& y : a)
            if (&x != &y && y.at >= 0 && x.at < y.at + y.bytes && y.at < x.at + x.bytes) {
                printf("FAIL %s and %s overlap (n=%d m=%d tables=%d wide=%d use=%d)\n", x.name, y.name, n, m, tables, wide, use);
                return false;
            }
    }
    if (!wide && (L.off_unsat < 0 || L.off_tau < 0 || L.off_cut < 0 || L.cuts < 1)) { printf("FAIL lazy arrays\n"); return false; }
    if ((thr && L.off_thr < 0) || (st && L.off_st < 0)) { printf("FAIL thr or state\n"); return false; }
    if (!wide && L.off_cnt + pad4(nl) * 16 + 31 * 64 > L.total) { printf("FAIL counts read past the total\n"); return false; }
    const int end = thr ? L.off_thr : L.total;
    if (tight && (L.off_queue != L.off_sw || L.off_flips != -1 || st || wide || end - L.off_sw < warps * kQueue * 4)) { printf("FAIL tight\n"); return false; }
    return L.total % 16 == 0;
}

static int random_layouts(int cases) {
    long tights = 0, few_cuts = 0;
    for (int c = 0; c < cases; ++c) {
        const bool wide = rnd() % 3 == 0, adapt = rnd() & 1, st = rnd() & 1, serve = rnd() & 1;
        const int use = serve ? kServe : kTable;
        const int n = in(500, 12000), m = in(std::max(4, n / 64), n), dv = wide ? in(16, 64) : in(1, 15), dc = in(2, 64), P = in(0, 3), warps = 4 << in(0, 3);
        const SmemLayout A = smem_layout(n, m, 100, dv, dc, adapt, st, P);
        if (!sane(A, n, m, n, dv, dc, adapt, st, P, dv > kNarrowDegree, kLaunch, warps)) return 1;
        if (!st && dv <= kNarrowDegree && n >= 500) {
            const SmemLayout B = smem_layout(n, m, 100, dv, dc, adapt, false, kTight, -1, -1, kLaunch, warps);
            if (!sane(B, n, m, n, dv, dc, adapt, false, kTight, false, kLaunch, warps)) return 1;
        }
        const int C = 1 << in(0, 3), nl = C > 1 && !serve ? split_local_max(n, C) : n, bytes = in(30000, 232448);
        int tb = -1;
        const SmemLayout J = job_layout(n, m, 100, dv, dc, adapt, st, wide, P, nl, bytes, &tb, use, warps);
        if (!sane(J, n, m, nl, dv, dc, adapt, st, tb, wide, use, warps)) return 1;
        if ((tb & ~(P | kTight)) || ((tb & kTight) && (st || wide))) { printf("FAIL placement %d of %d\n", tb, P); return 1; }
        if (serve && !wide && (J.cuts < 1 || J.cuts > kChain || (st && J.total <= bytes && J.cuts != kChain))) {
            printf("FAIL %d cutoff tables\n", J.cuts);
            return 1;
        }
        if (J.total <= bytes) {
            tights += tb == kTight;
            few_cuts += serve && !wide && J.cuts < kChain;
            // a job no larger fits as well, whatever the tables
            const int n2 = in(std::max(8, n / 2), n), m2 = in(std::max(4, n2 / 64), std::max(std::max(4, n2 / 64), std::min(m, n2)));
            if (C == 1 && m2 <= m) {
                const SmemLayout S = job_layout(n2, m2, 100, dv, dc, adapt, st, wide, P, n2, J.total, &tb, use, warps);
                if (S.total > J.total) { printf("FAIL smaller job: %d > %d\n", S.total, J.total); return 1; }
                if (!sane(S, n2, m2, n2, dv, dc, adapt, st, tb, wide, use, warps)) return 1;
            }
        }
    }
    printf("ok %d %ld %ld\n", cases, tights, few_cuts);
    return 0;
}

// The former bytes of a code without its state or tables, and whether the present ones fit.
static int limits() {
    const int optin = 232448;
    long held = 0;
    for (int use : {kLaunch, kTable, kServe})
        for (int dv : {1, 3, 7, 8, 15, 16, 40})
            for (int adapt = 0; adapt < 2; ++adapt)
                for (int n = 5000; n < 11400; n += n < 5400 || n > 9900 ? 1 : 37)
                    for (int m = std::max((n + 63) / 64, dv); m < n; m += m < 1300 ? 1 + m / 64 : m / 8) {
                        const bool was_wide = dv > 7, wide = dv > kNarrowDegree;
                        const int was_static = use == kLaunch ? 0 : use == kTable ? 248 : 1984;
                        const int was = 5408 + pad4(n) * (was_wide ? 32 : 16) + pad4(n + 1) * 4 +
                                        ((m + 1) * (was_wide ? 4 : 16) + 15) / 16 * 16 + (adapt ? 2048 : 0);
                        if (was > optin - was_static) continue;
                        ++held;
                        const int now_static = use == kLaunch ? 0 : use == kTable ? (int)sizeof(Job) + 16 : (int)sizeof(ServeShared);
                        int tb = 0;
                        const int now = use == kLaunch
                            ? std::min(smem_layout(n, m, 100, dv, 64, adapt, false, 0).total,
                                       wide ? 1 << 30 : smem_layout(n, m, 100, dv, 64, adapt, false, kTight).total)
                            : job_layout(n, m, 100, dv, 64, adapt, false, wide, 0, n, optin - now_static, &tb, use).total;
                        if (now > optin - now_static) {
                            printf("FAIL use %d: n=%d m=%d degree %d adapt %d was %d of %d, now %d of %d\n", use, n, m, dv, adapt, was,
                                   optin - was_static, now, optin - now_static);
                            return 1;
                        }
                    }
    printf("ok %ld\n", held);
    return 0;
}

int main(int argc, char** argv) {
    if (argc < 3) return limits();
    s = strtoull(argv[1], nullptr, 10);
    return random_layouts(atoi(argv[2]));
}
"""


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    nvcc = _build.nvcc()
    if shutil.which(nvcc) is None and not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("layout_lazy")
    src, exe = d / "layout_lazy.cu", d / "layout_lazy"
    src.write_text(SRC)
    subprocess.check_call([nvcc, "-std=c++17", "-O1", "-I", _build.CSRC, "-gencode", "arch=compute_103a,code=sm_103a",
                           "-o", str(exe), str(src)])
    return str(exe)


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_arrays_of_random_layouts(prog, seed):
    out = subprocess.run([prog, str(seed), "20000"], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout + out.stderr
    tag, cases, tights, few_cuts = out.stdout.split()
    assert tag == "ok" and int(cases) == 20000 and int(tights) > 0 and int(few_cuts) > 0


def test_no_code_that_fitted_is_refused(prog):
    """A single launch, a job of a table and a request to the server, with every adjacency table and
    the state out of shared memory, on a device of 227 KB per block."""
    out = subprocess.run([prog], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
    assert out.stdout.startswith("ok") and int(out.stdout.split()[1]) > 100000
