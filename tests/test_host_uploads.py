"""Bytes that a call copies to the device stay as they are until the stream has been waited
for: a copy from pageable memory may read them after the call that queued it.  The library's
host code runs on the CPU here, linked against a stand-in runtime (fake_cudart.c) whose
device memory is host memory and whose kernels do nothing; it compares every source when it
is queued and when the stream is waited for, with freed memory overwritten."""
import ctypes
import glob
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

P, I64, I32 = ctypes.c_void_p, ctypes.c_int64, ctypes.c_int


def _calls(path):
    """Runs in a process of its own: every kind of product once; returns the two counts."""
    lib = ctypes.CDLL(path)
    nul = (ctypes.c_char * (1 << 16))()   # an empty operand's arrays

    class Opts(ctypes.Structure):
        _fields_ = [("f", I32 * 6), ("margin", ctypes.c_float), ("g", I32 * 8)]

    def opts(**kw):
        o = Opts()
        lib.spgemm_opts_default(ctypes.byref(o))
        if kw.get("predictor"):
            o.f[0] = 1
        if kw.get("esc"):
            o.g[1] = 1
        return ctypes.byref(o)

    def ok(status):
        assert status == 0, status

    ctx, merge = P(), P()
    ok(lib.spgemm_ctx_create(ctypes.byref(ctx), None, None, None, None))
    ok(lib.spgemm_ctx_create(ctypes.byref(merge), None, None, None, None))

    def mat(make=lib.spgemm_mat_csc, n=1000, nnz=0):
        h = P()
        ok(make(ctx, ctypes.byref(h), I64(n), I64(n), I64(nnz), nul, nul, nul, 0))
        return h

    out = P()
    ok(lib.spgemm_multiply(ctx, mat(), mat(lib.spgemm_mat_csr), 0, None, ctypes.byref(out)))
    for count in (1, 2, 300):
        As, Bs, Cs = (P * count)(*[mat() for _ in range(count)]), (P * count)(*[mat() for _ in range(count)]), (P * count)()
        ok(lib.spgemm_batch(ctx, count, As, Bs, 0, None, Cs))
        plan = P()
        ok(lib.spgemm_batch_plan(ctx, count, As, Bs, 0, None, ctypes.byref(plan)))
        ok(lib.spgemm_batch_execute(plan))
        ok(lib.spgemm_plan_destroy(plan))
    ok(lib.spgemm_predictor_set(ctx, nul))
    ok(lib.spgemm_batch(ctx, 2, As, Bs, 0, opts(predictor=True), Cs))
    ok(lib.spgemm_summa_blocked(ctx, mat(), mat(), 3, 0, None, ctypes.byref(out)))
    ok(lib.spgemm_summa_blocked(ctx, mat(), mat(), 3, 0, opts(esc=True), ctypes.byref(out)))
    ok(lib.spgemm_summa_pipelined(ctx, merge, mat(), mat(), 3, 0, None, ctypes.byref(out)))
    D = P()
    ok(lib.spgemm_mat_to_dcsc(ctx, mat(), 1, ctypes.byref(D)))
    ok(lib.spgemm_multiply(ctx, D, D, 0, None, ctypes.byref(out)))
    ok(lib.spgemm_ctx_destroy(ctx))
    ok(lib.spgemm_ctx_destroy(merge))
    return lib.fake_copies(), lib.fake_stale()


@pytest.fixture(scope="module")
def host_lib(tmp_path_factory):
    from paper_1006_2183_gb300 import build
    build.build()
    path = str(tmp_path_factory.mktemp("host") / "libhost.so")
    fake = path + ".o"
    objs = [os.path.join(build.OUT_DIR, os.path.basename(s) + ".o") for s in glob.glob(os.path.join(build.CSRC, "*.cu"))]
    subprocess.run(["gcc", "-O1", "-fPIC", "-c", os.path.join(HERE, "fake_cudart.c"), "-o", fake], check=True)
    subprocess.run(["g++", "-shared", "-fPIC", "-o", path, *objs, fake, "-lpthread"], check=True)
    return path


def test_sources_of_copies_last_until_the_wait(host_lib):
    env = dict(os.environ, MALLOC_PERTURB_="85", MALLOC_TRIM_THRESHOLD_=str(1 << 30), MALLOC_MMAP_THRESHOLD_=str(1 << 30))
    r = subprocess.run([sys.executable, os.path.abspath(__file__), host_lib], env=env, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr
    copies, stale = map(int, r.stdout.split())
    assert copies > 0
    assert stale == 0, f"{stale} of {copies} copies read memory that was given up before the wait"


if __name__ == "__main__":
    print(*_calls(sys.argv[1]))
