"""Solves on several streams and host threads at once, and on a stream that owns only some of
the GPU's SMs (a green context): the CG's cooperative launch takes as many CTAs as the stream's
SMs hold, or its passes go in separate launches.  Every form gives the bits of the solve alone."""
import ctypes as C
import math
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (kind, d, M, N, Q, precision): rows that stay in shared memory, several queries, FP64, rows
# that stream (one query), and more queries than the cooperative loop takes
SHAPES = [("ac_manufactured", 64, 512, 4, 1, "fp32"),
          ("logistic_grad", 700, 3001, 3, 1, "fp32"),
          ("ac_manufactured", 130, 700, 3, 5, "fp64"),
          ("logistic_grad", 2003, 9001, 2, 1, "fp32"),
          ("ac_manufactured", 101, 503, 2, 65, "fp32")]


def _solver(shape, seed):
    from paper_2510_02635_gb300 import fbsde as fb
    kind, d, M, N, Q, prec = shape
    sigma, T = (float(d), 1.0) if kind == "logistic_grad" else (1.0, 0.5)
    solver = fb.Solver(kind, d, N, M, sigma, T, Q=Q, precision=prec, cg_max_iter=1000,
                       cg_tol=1e-12 if prec == "fp64" else 1e-6)
    x0 = np.random.default_rng(seed).standard_normal((Q, d)) / math.sqrt(d)
    return solver, torch.tensor(x0, device="cuda")


def test_threads_and_streams_at_once_give_the_bits_of_each_alone():
    jobs = [(*_solver(shape, i), i) for i, shape in enumerate(SHAPES)]
    ref = [solver.solve(x0, seed=seed) for solver, x0, seed in jobs]
    torch.cuda.synchronize()
    got, failed = [[] for _ in jobs], []

    def work(i):
        try:
            solver, x0, seed = jobs[i]
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(4):
                    got[i].append(solver.solve(x0, seed=seed))
                torch.cuda.current_stream().synchronize()
        except BaseException as exc:   # reported by the test's own thread
            failed.append((i, exc))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for r, outs in zip(ref, got):
        assert len(outs) == 4
        for out in outs:
            assert out["status"] == 0
            assert torch.equal(out["u0"], r["u0"]) and torch.equal(out["grad"], r["grad"])


def _green_stream(sms):
    """A stream on a green context of about `sms` SMs, and its SM count (driver API; a
    CUdevResource has 144 bytes, its SM count at offset 96)."""
    cu = C.CDLL("libcuda.so.1")

    def call(name, *args):
        st = getattr(cu, name)(*args)
        assert st == 0, (name, st)

    torch.cuda.synchronize()
    dev, groups = C.c_int(), C.c_uint(1)
    whole, part = C.create_string_buffer(144), C.create_string_buffer(144)
    rest = C.create_string_buffer(144)
    desc, ctx, stream = C.c_void_p(), C.c_void_p(), C.c_void_p()
    call("cuDeviceGet", C.byref(dev), torch.cuda.current_device())
    call("cuDeviceGetDevResource", dev, whole, 1)
    call("cuDevSmResourceSplitByCount", part, C.byref(groups), whole, rest, 0, sms)
    call("cuDevResourceGenerateDesc", C.byref(desc), part, 1)
    call("cuGreenCtxCreate", C.byref(ctx), desc, dev, 1)
    call("cuGreenCtxStreamCreate", C.byref(stream), ctx, 1, 0)
    return cu, ctx, stream, int.from_bytes(part.raw[96:100], "little")


def test_stream_of_a_few_sms_gives_the_same_bits():
    cu, ctx, stream, sms = _green_stream(16)
    assert 16 <= sms < torch.cuda.get_device_properties(0).multi_processor_count
    ext = torch.cuda.ExternalStream(stream.value)
    try:
        for i, shape in enumerate(SHAPES):
            solver, x0 = _solver(shape, i)
            ref = solver.solve(x0, seed=i)
            torch.cuda.synchronize()
            with torch.cuda.stream(ext):
                out = solver.solve(x0, seed=i)
                ext.synchronize()
            assert out["status"] == 0
            assert torch.equal(out["u0"], ref["u0"]) and torch.equal(out["grad"], ref["grad"])
    finally:
        torch.cuda.synchronize()
        cu.cuStreamDestroy_v2(stream)
        cu.cuGreenCtxDestroy(ctx)
