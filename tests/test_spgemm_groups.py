"""The row products of the setup's SpGEMM by groups of lanes, on the CPU.

csrc/spgemm_groups.cuh is compiled for the host and its warps run in lockstep,
a fiber a lane that hands over at every warp operation.  Every group and table
size, the one-run form (rows into a temporary) and the two-run form (count, then
write in place) give the serial product bit for bit, rows of more columns than
the table are handed on and not written, and no table ever holds more keys than
its columns and one step of its group.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2001_05798_gb300", "csrc")

HOST = r"""
#include <cstddef>
#include <cstdint>
#include <cstring>
#include <ucontext.h>
#define __global__ static
#define __device__ static
#define __forceinline__ inline
#define __launch_bounds__(x)
#define __shared__
struct int4 { int x, y, z, w; };
static int4 make_int4(int x, int y, int z, int w) { return int4{x, y, z, w}; }
struct Dim { unsigned x; };
static Dim threadIdx, blockIdx, gridDim;
alignas(16) static double mem[1 << 13];
#define sgg_mem mem
static ucontext_t home, lanes[32];
static char stacks[32][1 << 16];
static bool alive[32];
static int cur, warp0, diverged, peak;
static long seq[32];
static uint64_t box[32];
static void yield() { swapcontext(&lanes[cur], &home); }
static void meet()
{
    ++seq[cur];
    yield();
    for (int l = 0; l < 32; ++l)
        if (seq[l] != seq[cur]) diverged = 1;
}
static void __syncwarp() { meet(); yield(); }
template <class T> static T __shfl_sync(unsigned, T v, int src, int width = 32)
{
    T r;
    memcpy(&box[cur], &v, sizeof v);
    meet();
    memcpy(&r, &box[(cur & ~(width - 1)) + (src & (width - 1))], sizeof r);
    yield();
    return r;
}
static unsigned __ballot_sync(unsigned, bool p)
{
    box[cur] = p;
    meet();
    unsigned m = 0;
    for (int l = 0; l < 32; ++l) m |= (unsigned)(box[l] != 0) << l;
    yield();
    return m;
}
static bool __any_sync(unsigned m, bool p) { return __ballot_sync(m, p) != 0; }
static double __dadd_rn(double a, double b) { return a + b; }
static double __dmul_rn(double a, double b) { return a * b; }
static int atomicCAS(int *p, int c, int v) { const int o = *p; if (o == c) *p = v; return o; }
static int atomicAdd(int *p, int v)
{
    const int o = *p;
    *p += v;
    if ((char *)p >= (char *)mem && (char *)p < (char *)(mem + (1 << 13)) && *p > peak) peak = *p;
    return o;
}
static int min(int a, int b) { return a < b ? a : b; }
#include "body.inc"
struct Args { int nr; const int *lrp, *lci; const double *lv; const int *rrp, *rci; const double *rv; const int *crp;
              int *cnt, *oci; double *ov; int *long_rows, *nlong; };
static Args A;
static int form;
static void lane_main()
{
    using namespace gw;
#define RUN(k, G, CAP) \
    if (form == k) k_sgg<G, CAP>(A.nr, A.lrp, A.lci, A.lv, A.rrp, A.rci, A.rv, A.crp, A.cnt, A.oci, A.ov, A.long_rows, A.nlong);
    RUN(0, 4, 16) RUN(1, 4, 64) RUN(2, 8, 64) RUN(3, 16, 64) RUN(4, 16, 128) RUN(5, 32, 128)
    alive[cur] = false;
    for (;;) yield();
}
extern "C" int run(int f, int blocks, int nr, const int *lrp, const int *lci, const double *lv, const int *rrp,
                   const int *rci, const double *rv, const int *crp, int *cnt, int *oci, double *ov, int *long_rows,
                   int *nlong, int *peak_out)
{
    A = Args{nr, lrp, lci, lv, rrp, rci, rv, crp, cnt, oci, ov, long_rows, nlong};
    form = f, diverged = 0, peak = 0, gridDim.x = (unsigned)blocks;
    for (int b = 0; b < blocks; ++b)
        for (int w = 0; w < gw::SGG_BS / 32; ++w) {
            for (int l = 0; l < 32; ++l) {
                getcontext(&lanes[l]);
                lanes[l].uc_stack.ss_sp = stacks[l];
                lanes[l].uc_stack.ss_size = sizeof stacks[l];
                lanes[l].uc_link = nullptr;
                makecontext(&lanes[l], lane_main, 0);
                alive[l] = true, seq[l] = 0;
            }
            for (bool any = true; any;) {
                any = false;
                for (cur = 0; cur < 32; ++cur)
                    if (alive[cur]) {
                        threadIdx.x = (unsigned)(w * 32 + cur), blockIdx.x = (unsigned)b;
                        swapcontext(&home, &lanes[cur]);
                        any |= alive[cur];
                    }
            }
        }
    *peak_out = peak;
    return diverged;
}
"""

# (lanes a row, columns of the table); the index is the form number above
FORMS = [(4, 16), (4, 64), (8, 64), (16, 64), (16, 128), (32, 128)]


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("sgg")
    body = open(os.path.join(CSRC, "spgemm_groups.cuh")).read().replace("#pragma once", "")
    (d / "body.inc").write_text(body.replace("extern __shared__ double sgg_mem[];", ""))
    (d / "host.cpp").write_text(HOST)
    so = str(d / "host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-w", "-shared", "-fPIC", "-I", str(d),
                    str(d / "host.cpp"), "-o", so], check=True, capture_output=True, text=True)
    return ctypes.CDLL(so)


def csr(rows):
    """rows: a list of lists of (column, value)."""
    rp = np.zeros(len(rows) + 1, np.int32)
    rp[1:] = np.cumsum([len(r) for r in rows])
    ci = np.array([c for r in rows for c, _ in r] or [0], np.int32)
    v = np.array([x for r in rows for _, x in r] or [0.0], np.float64)
    return rp, ci, v


def serial(L, R):
    out = []
    for e0, e1 in zip(L[0][:-1], L[0][1:]):
        acc = {}
        for e in range(e0, e1):
            k = L[1][e]
            for f in range(R[0][k], R[0][k + 1]):
                acc[int(R[1][f])] = acc.get(int(R[1][f]), 0.0) + L[2][e] * R[2][f]
        out.append(sorted(acc.items()))
    return out


def check(host, form, L, R):
    G, cap = FORMS[form]
    nr = len(L[0]) - 1
    ref = serial(L, R)
    ptr = lambda a: None if a is None else a.ctypes.data_as(ctypes.c_void_p)

    def run(crp, cnt, oci, ov):
        long_rows, nlong, peak = np.full(nr, -1, np.int32), np.zeros(1, np.int32), ctypes.c_int()
        diverged = host.run(form, 2, nr, *[ptr(a) for a in (*L, *R)], ptr(crp), ptr(cnt), ptr(oci), ptr(ov),
                            ptr(long_rows), ptr(nlong), ctypes.byref(peak))
        assert not diverged
        assert peak.value <= cap + G, (peak.value, cap, G)
        return sorted(long_rows[:nlong[0]].tolist())

    over = [i for i, r in enumerate(ref) if len(r) > cap]
    counts = np.array([0 if len(r) > cap else len(r) for r in ref], np.int32)
    full = np.array([len(r) for r in ref], np.int32)
    crp = np.zeros(nr + 1, np.int32)
    crp[1:] = np.cumsum(full)
    # one run: every row in its cap entries of the temporary
    cnt, tci, tcv = np.full(nr, -7, np.int32), np.full(nr * cap, -1, np.int32), np.zeros(nr * cap)
    assert run(None, cnt, tci, tcv) == over
    assert np.array_equal(cnt, counts)
    # two runs: count only, then in place
    cnt2 = np.full(nr, -7, np.int32)
    assert run(None, cnt2, None, None) == over
    assert np.array_equal(cnt2, counts)
    oci, ov = np.full(max(1, crp[-1]), -1, np.int32), np.zeros(max(1, crp[-1]))
    assert run(crp, None, oci, ov) == []
    for i, r in enumerate(ref):
        cols = np.array([c for c, _ in r], np.int32)
        vals = np.array([x for _, x in r])
        if len(r) > cap:
            assert (oci[crp[i]:crp[i + 1]] == -1).all()
            continue
        for ci, v, o in ((tci, tcv, i * cap), (oci, ov, crp[i])):
            assert np.array_equal(ci[o:o + len(r)], cols), i
            assert np.array_equal(v[o:o + len(r)].view(np.uint64), vals.view(np.uint64)), i


@pytest.mark.parametrize("form", range(len(FORMS)))
def test_random_products(host, form):
    """Rows from empty to past the table, lists shorter and longer than the
    group, a last warp with idle groups."""
    G, cap = FORMS[form]
    rng = np.random.default_rng(form)
    nmid, ncol = 40, 3 * cap

    def rows(n, nc, lens):
        return [[(int(c), float(rng.standard_normal())) for c in sorted(rng.choice(nc, min(nc, k), replace=False))]
                for k in rng.choice(lens, n)]

    R = csr(rows(nmid, ncol, [0, 1, G - 1, G, G + 1, 2 * G + 1]))
    check(host, form, csr(rows(37, nmid, [0, 1, 2, 3, G, G + 3, 2 * G + 1])), R)


@pytest.mark.parametrize("form", range(len(FORMS)))
def test_a_full_row_stops(host, form):
    """A row that passes its table beside rows of the same warp that go on:
    it inserts no more columns while it waits for them."""
    G, cap = FORMS[form]
    # right rows 0 .. 31: G columns each, all distinct; right row 32: one column
    R = csr([[(G * k + c, 1.0 + k) for c in range(G)] for k in range(32)] + [[(5, 2.0)]] * 33)
    wide = [(k, 0.5) for k in range(32)]
    narrow = [(32 + k, 0.25) for k in range(33)]
    check(host, form, csr([wide, narrow, narrow, wide, narrow, wide, wide, narrow]), R)
