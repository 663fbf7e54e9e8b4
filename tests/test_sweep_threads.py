"""Sweeps of two contexts on two host threads at once: each keeps its own precision,
scratch and streams.  Without a GPU on the host build of the sweeps, with one on the
library itself."""
import ctypes
import os
import shutil
import subprocess
import threading

import numpy as np
import pytest

from oracle import rgf
from paper_2601_04904_gb300 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


def test_host_sweeps_in_two_precisions_at_once(tmp_path):
    """FP64 solves on one thread give their bits while another thread's sweeps ask for
    tensor-core products, and every one of those asks."""
    gxx = shutil.which("g++")
    if not gxx or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    out = tmp_path / "two_threads.so"
    subprocess.run([gxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-x", "c++",
                    os.path.join(ROOT, "tests", "host_sweep", "two_threads.cpp"), "-I", CUDA_INC, "-o", str(out)],
                   check=True)
    lib = ctypes.CDLL(str(out))
    sizes, a = [4] * 40, 2
    A = rgf.assemble_a(inputs.hamiltonian_sizes(sizes, a), 0.3, 1e-3, 0.5)
    B = inputs.lesser_rhs_sizes(sizes, a)
    fa, fb = inputs.pack_sizes(A), inputs.pack_sizes(B)
    ptrs = lambda f: (ctypes.c_void_p * 6)(*[f[k].ctypes.data for k in inputs.KEYS])

    def solve():
        r, l = ({k: np.zeros_like(v) for k, v in fa.items()} for _ in range(2))
        rc = lib.host_solve(len(sizes), (ctypes.c_int * len(sizes))(*sizes), a, 0, ptrs(fa), ptrs(fb), ptrs(r), ptrs(l))
        return rc, r, l

    _, r0, l0 = solve()
    bad, stop = [], threading.Event()

    def other():
        while not stop.is_set():
            if lib.host_tc_sweeps(2000) != 2000:
                bad.append("a sweep used another thread's precision")

    t = threading.Thread(target=other)
    t.start()
    try:
        for _ in range(100):
            rc, r, l = solve()
            assert rc == 0
            assert all((r[k] == r0[k]).all() and (l[k] == l0[k]).all() for k in inputs.KEYS)
    finally:
        stop.set()
        t.join()
    assert not bad


@pytest.mark.gpu
def test_contexts_on_their_own_threads_give_their_bits():
    """Solves of three contexts in different precisions, graphs and direct launches, at
    the same time on three host threads: bitwise those of a context alone."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_04904_gb300 import qsi

    work = []
    for prec, n, b, a, seed in ((qsi.FP64_EMU, 12, 72, 20, 1), (qsi.FP64, 6, 40, 8, 2), (qsi.MIXED, 8, 130, 0, 3)):
        stream = torch.cuda.Stream()
        ctx = qsi.Context(0, stream=stream)
        H, A = qsi.to_device(inputs.hamiltonian(n, b, a, seed=seed)), qsi.device_zeros(n, b, a)
        B = qsi.to_device(inputs.lesser_rhs(n, b, a, seed=seed + 10))
        torch.cuda.synchronize()
        ctx.assemble(H, 0.3, 1e-3, 0.5, out=A)
        ctx.synchronize()
        work.append((ctx, A, B, prec, (n, b, a)))

    def passes(w, count, out):
        ctx, A, B, prec, shape = w
        try:
            for _ in range(count):
                GR, GL, R, L = (qsi.device_zeros(*shape) for _ in range(4))
                torch.cuda.current_stream().synchronize()  # their zeros are written on torch's stream
                for _ in range(3):  # the first call solves directly and captures, the others replay
                    ctx.solve(A, [B], GR, [GL], precision=prec)
                f = ctx.factor(A, B, prec)
                ctx.selquad(f, R, L)
                ctx.synchronize()
                f.close()
                out.append((GR, GL, R, L))
        except Exception as e:  # reported by the main thread
            out.append(e)

    alone = []
    for w in work:
        passes(w, 1, alone)
    together = [[] for _ in work]
    threads = [threading.Thread(target=passes, args=(w, 6, o)) for w, o in zip(work, together)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for ref, got in zip(alone, together):
        assert len(got) == 6
        for g in got:
            assert not isinstance(g, Exception), g
            for x, y in zip(ref, g):
                for k in qsi.KEYS:
                    assert (x[k] == y[k]).all(), k
    for w in work:
        w[0].close()
