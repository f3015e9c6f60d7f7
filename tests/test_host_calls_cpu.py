"""The CUDA runtime calls that the host side makes, checked without a GPU.

libkgrape.so runs in a child process with a stand-in for the runtime calls it makes (LD_PRELOAD): nothing
is executed, every call is written down, and one launch can be made to fail.
"""
import json
import os
import shutil
import subprocess
import sys

import pytest

from paper_2010_03598_gb300 import _abi
from paper_2010_03598_gb300 import build as kbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = "/usr/local/cuda"

FAKE = r"""
#include <cuda_runtime_api.h>
#include <stdarg.h>
#include <stdio.h>
#include <stdlib.h>
static FILE* out;
static long handles = 1, launches = 0;
static void note(const char* fmt, ...) {
  va_list ap;
  if (!out) out = fopen(getenv("FAKE_LOG"), "w");
  va_start(ap, fmt); vfprintf(out, fmt, ap); va_end(ap);
  fflush(out);
}
static cudaError_t launch(const void* fn, size_t smem, cudaStream_t s) {
  const char* f = getenv("FAKE_FAIL");
  const int bad = f && atol(f) == launches;
  ++launches;
  note("launch %p %zu %p %d\n", fn, smem, (void*)s, bad);
  return bad ? cudaErrorInvalidValue : cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* fn, enum cudaFuncAttribute a, int v) { note("attr %p %d\n", fn, v); return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* fn, int t, size_t s) { *n = 1; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* fn, int t, size_t s, unsigned f) { *n = 1; return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)200 << 30; return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind k) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f) { *s = (cudaStream_t)(handles++ << 8); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned f) { *e = (cudaEvent_t)(handles++ << 8); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { note("record %p %p\n", (void*)e, (void*)s); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) { note("wait %p %p\n", (void*)s, (void*)e); return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void* fn, dim3 g, dim3 b, void** a, size_t m, cudaStream_t s) { return launch(fn, m, s); }
cudaError_t cudaLaunchCooperativeKernel(const void* fn, dim3 g, dim3 b, void** a, size_t m, cudaStream_t s) { return launch(fn, m, s); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void** a) { return launch(fn, c->dynamicSmemBytes, c->stream); }
"""

PRELUDE = r"""
import ctypes, json, sys
sys.path.insert(0, {root!r})
from paper_2010_03598_gb300 import _abi as a
lib = a.lib()
WS = ctypes.c_void_p(1 << 20)   # never dereferenced: no copy is executed
def chain(L): return a.KgChain(L, a.KG_HC_SX_SITE, 0, 0, 0, 1.0, 0.5, 1.0)
def opts(**k):
    o = dict(N=4, m=8, prec=a.KG_PREC_C64_F64REC, grad=a.KG_GRAD_CENTERED, ckpt_every=0, tile_bits=0, ctas=0, flags=0,
             dt=0.1, breakdown_tol=0.0, mem_budget=0)
    o.update(k)
    return a.KgOptions(**o)
P = ctypes.c_void_p(1 << 20)
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    gcc = shutil.which("gcc")
    if gcc is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime_api.h")):
        pytest.skip("needs a C compiler and the CUDA headers")
    if not os.path.exists(_abi.LIB_PATH):
        kbuild.build()
    d = tmp_path_factory.mktemp("fake")
    (d / "fake.c").write_text(FAKE)
    subprocess.run([gcc, "-shared", "-fPIC", "-O1", "-I", os.path.join(CUDA, "include"), str(d / "fake.c"), "-o",
                    str(d / "fake.so")], check=True)

    def run(code, fail=None):
        """The child's printed JSON and the calls it made, as lists of words."""
        log = d / "log"
        env = dict(os.environ, LD_PRELOAD=str(d / "fake.so"), FAKE_LOG=str(log))
        env.pop("FAKE_FAIL", None)
        if fail is not None:
            env["FAKE_FAIL"] = str(fail)
        log.write_text("")
        r = subprocess.run([sys.executable, "-c", PRELUDE.format(root=ROOT) + code], env=env, capture_output=True,
                           text=True, timeout=120)
        assert r.returncode == 0, r.stderr
        return json.loads(r.stdout), [line.split() for line in log.read_text().splitlines()]

    return run


# Launches of every kernel family at sizes whose shared memory differs.
LAUNCHES = r"""
n = 0
for prec in (a.KG_PREC_C64_F64REC, a.KG_PREC_C128):
    for L in (3, 6, 7, 8, 9, 10, 11, 12, 13, 16, 18, 20):
        for m in (1, 6, 13, 24, 32):
            for kw in (dict(), dict(tile_bits=6), dict(tile_bits=min(L, 10)), dict(flags=a.KG_FLAG_FULL_REORTH, tile_bits=min(L, 9))):
                if kw and m != 6: continue
                h = ctypes.c_void_p()
                c, o = chain(L), opts(m=m, prec=prec, **kw)
                a.check(lib.kg_create(ctypes.byref(h), c, o, WS, 1 << 50, None), "create")
                a.check(lib.kg_evaluate(h, P, P, P, P, P), "evaluate")
                lib.kg_destroy(h)
                n += 1
for prec in (a.KG_PREC_C64_F64REC, a.KG_PREC_C128, a.KG_PREC_FF):
    for L, K, p in ((8, 3, 1), (9, 3, -1), (10, 4, 1), (11, 4, 0), (14, 4, 1), (13, 6, 1), (17, 4, 1), (20, 4, 1), (14, 7, 0)):
        for nt in (0, 256, 512):
            h = ctypes.c_void_p()
            s, o = a.KgSector(L, K, p, nt, 0, 2.0, 1.0, 1.0), opts(prec=prec)
            st = lib.kg_sector_create(ctypes.byref(h), s, o, 2, WS, 1 << 50, None)
            if st == a.KG_ERR_INVALID_ARG: continue   # a block too small for the subspace
            a.check(st, "sector create")
            a.check(lib.kg_sector_evaluate(h, P, P, P, P, P), "sector evaluate")
            lib.kg_sector_destroy(h)
            n += 1
for m in (4, 24):
    B = 6
    cs = (a.KgChain * B)(*[chain(L) for L in (6, 9, 10, 12, 13, 16)])
    ptrs = (ctypes.c_void_p * B)(*[1 << 20] * B)
    h = ctypes.c_void_p()
    o = opts(m=m)
    a.check(lib.kg_batch_create(ctypes.byref(h), B, cs, o, None, ptrs, ptrs, ptrs, P, ptrs, WS, 1 << 50, None), "batch")
    a.check(lib.kg_batch_launch(h), "launch")
    lib.kg_batch_destroy(h)
    n += 1
print(json.dumps(n))
"""


def test_a_kernels_shared_memory_limit_does_not_depend_on_the_call(fake):
    # The limit is a property of the kernel in the whole process: a call that set it to its own size would
    # let another host thread's larger launch, between that thread's setting and launch, fail.
    n, calls = fake(LAUNCHES)
    limit = {}
    launched = 0
    for c in calls:
        if c[0] == "attr":
            limit.setdefault(c[1], set()).add(int(c[2]))
        elif c[0] == "launch":
            launched += 1
            assert int(c[2]) <= min(limit[c[1]]), c
    assert launched >= n > 100
    assert all(len(v) == 1 for v in limit.values()), {k: sorted(v) for k, v in limit.items() if len(v) > 1}


BATCH = r"""
B = 6
cs = (a.KgChain * B)(*[chain(L) for L in (6, 9, 10, 13, 14, 16)])
ptrs = (ctypes.c_void_p * B)(*[1 << 20] * B)
h = ctypes.c_void_p()
o = opts()
a.check(lib.kg_batch_create(ctypes.byref(h), B, cs, o, None, ptrs, ptrs, ptrs, P, ptrs, WS, 1 << 50, ctypes.c_void_p(0x77)), "batch")
print(json.dumps(lib.kg_batch_launch(h)))
"""


@pytest.mark.parametrize("fail", [None, 0, 1, 3, 5])
def test_a_batch_joins_its_streams_even_if_a_launch_fails(fake, fail):
    # One launch per chain length on a stream each; `fail` is the launch that the runtime refuses.  Whatever was
    # launched on a side stream has to be waited for by the caller's stream: it writes the caller's buffers.
    status, calls = fake(BATCH, fail)
    assert status == (_abi.KG_OK if fail is None else _abi.KG_ERR_CUDA)
    caller = "0x77"
    started = {c[3] for c in calls if c[0] == "launch" and c[4] == "0"}
    assert len(started) == (6 if fail is None else fail)
    forked = {c[1] for c in calls if c[0] == "wait" and c[1] != caller}
    for s in (started | forked) - {caller}:
        last = max(i for i, c in enumerate(calls) if (c[0] == "launch" and c[3] == s) or (c[0] == "wait" and c[1] == s))
        events = {c[1]: i for i, c in enumerate(calls) if c[0] == "record" and c[2] == s and i > last}
        assert any(c[0] == "wait" and c[1] == caller and i > events.get(c[2], len(calls)) for i, c in enumerate(calls)), s
