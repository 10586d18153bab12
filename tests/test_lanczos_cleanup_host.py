"""What a Lanczos solve creates in the CUDA runtime (events, the capture's stream,
graphs) is given back on every way out of it: the library runs in a child process
against a stand-in for the runtime, on the CPU, whose kernels do nothing and whose
n-th call fails, for every n."""
import os
import subprocess
import sys

import pytest

from conftest import ROOT

FAKE = r"""
#include <stdlib.h>
#include <string.h>
static int calls, fail_at, live[3], made_streams;
static int err(void) { return ++calls == fail_at ? 999 : 0; }
#define F(name, args) int name args { return err(); }
void fake_reset(int n) { calls = 0; fail_at = n; made_streams = 0; }
int fake_calls(void) { return calls; }
int fake_live(int kind) { return live[kind]; }
int fake_streams(void) { return made_streams; }
static int make(void **p, int kind) { int e = err(); *p = e ? 0 : malloc(8); live[kind] += !e; return e; }
static int drop(void *p, int kind) { if (p) { free(p); --live[kind]; } return 0; }
int cudaMalloc(void **p, size_t n) { int e = err(); *p = e ? 0 : calloc(n + 256, 1); return e; }
int cudaFree(void *p) { free(p); return 0; }
int cudaMemcpy(void *d, const void *s, size_t n, int k) { int e = err(); if (!e) memcpy(d, s, n); return e; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int k, void *st) { int e = err(); if (!e) memcpy(d, s, n); return e; }
int cudaMemset(void *d, int v, size_t n) { int e = err(); if (!e) memset(d, v, n); return e; }
int cudaMemsetAsync(void *d, int v, size_t n, void *st) { int e = err(); if (!e) memset(d, v, n); return e; }
int cudaMemcpyFromSymbol(void *d, const void *s, size_t n, size_t o, int k) { memset(d, 0, n); return 0; }
int cudaMemcpyToSymbol(const void *d, const void *s, size_t n, size_t o, int k) { return 0; }
int cudaGetSymbolAddress(void **p, const void *s) { static char b[64]; *p = b; return 0; }
int cudaMemGetInfo(size_t *f, size_t *t) { *f = *t = (size_t)1 << 37; return err(); }
int cudaDeviceGetAttribute(int *v, int a, int d) {
    *v = a == 16 ? 152 : a == 95 ? 1 : a == 97 ? 232448 : 0;   /* multiprocessors, cooperative launch, shared memory */
    return err();
}
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaSetDevice(int d) { return 0; }
int cudaGetLastError(void) { return 0; }
const char *cudaGetErrorString(int e) { return "stand-in"; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int b, size_t s, unsigned fl) { *n = 1; return err(); }
F(cudaFuncSetAttribute, (const void *f, int a, int v))
F(cudaEventRecord, (void *e, void *s))
F(cudaEventSynchronize, (void *e))
int cudaEventElapsedTime(float *ms, void *a, void *b) { *ms = 1; return 0; }
int cudaEventCreate(void **e) { return make(e, 0); }
int cudaEventDestroy(void *e) { return drop(e, 0); }
int cudaStreamCreateWithFlags(void **s, unsigned f) { ++made_streams; return make(s, 1); }
int cudaStreamDestroy(void *s) { return drop(s, 1); }
F(cudaStreamSynchronize, (void *s))
F(cudaStreamBeginCapture, (void *s, int m))
int cudaStreamEndCapture(void *s, void **g) { return make(g, 2); }
int cudaGraphDestroy(void *g) { return drop(g, 2); }
int cudaGraphInstantiate(void **x, void *g, unsigned long long f) { return make(x, 2); }
int cudaGraphExecDestroy(void *x) { return drop(x, 2); }
F(cudaGraphLaunch, (void *x, void *s))
F(cudaLaunchCooperativeKernel, (const void *f, long long g0, int g1, long long b0, int b1, void **a, size_t s, void *st))
int __cudaLaunchKernel(void *k, long long g0, int g1, long long b0, int b1, void **a, size_t s, void *st) { return 0; }
int __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return 0; }
int __cudaPushCallConfiguration() { return 0; }
int __cudaPopCallConfiguration() { return 0; }
void **__cudaRegisterFatBinary(void *f) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) {}
void __cudaUnregisterFatBinary(void **h) {}
void __cudaRegisterFunction() {}
void __cudaRegisterVar() {}
"""

CHILD = r"""
import ctypes as C
import sys
import numpy as np
import paper_2203_04158_gb300 as G
from paper_2203_04158_gb300 import gbrank as B
fake = C.CDLL(sys.argv[1])
reorth, graph, profile = (int(v) for v in sys.argv[2:5])
L = 4
h = np.diag(np.full(L - 1, -1.0), 1)
h = h + h.T
lib = B.lib()
fake.fake_reset(0)
def solve():
    H = G.gbr_ham_create(L, h, np.full(L, 4.0), 2, 2)
    fake.fake_reset(n)
    o, r = B.LanczosOpts(20, reorth, G.GBR_PREC_FP64, 0, 0, graph, profile, 0.0, 0.0), B.LanczosResult()
    v, a, b = np.ones(36), np.zeros(20), np.zeros(20)
    p = lambda x: C.c_void_p(x.ctypes.data)
    rc = lib.gbr_lanczos(H, C.byref(o), p(v), C.byref(r), p(a), p(b), None, None)
    seen = fake.fake_calls()
    H.close()
    return rc, seen
n = 0
rc, total = solve()
print("plain", rc, total, fake.fake_streams())
failed, left = 0, []
for n in range(1, total + 1):
    rc, _ = solve()
    failed += rc != 0
    now = [fake.fake_live(k) for k in range(3)]
    if any(now):
        left.append((n, now))
        break
print("failed", failed, "left", left)
"""


@pytest.mark.parametrize("reorth,graph,profile", [(1, 0, 0), (1, 1, 0), (0, 1, 0), (0, 0, 1), (1, 0, 1)])
def test_every_failing_runtime_call_leaves_nothing_behind(tmp_path, reorth, graph, profile):
    import __graft_entry__
    __graft_entry__.build()
    src, so = tmp_path / "fake.c", tmp_path / "fake.so"
    src.write_text(FAKE)
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-w", "-o", str(so), str(src)])
    out = subprocess.check_output([sys.executable, "-c", CHILD, str(so), str(reorth), str(graph), str(profile)], cwd=ROOT,
                                  env=dict(os.environ, LD_PRELOAD=str(so), PYTHONPATH=ROOT), text=True, timeout=300)
    plain, fails = out.splitlines()[-2:]
    _, rc, total, streams = plain.split()
    assert int(rc) == 0 and int(total) > 20
    # a solve that runs in one launch captures nothing
    assert int(streams) == (1 if graph and not reorth else 0)
    assert fails.endswith("left []") and int(fails.split()[1]) > 10, fails
