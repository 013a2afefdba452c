"""Device memory: the fixed-point copies are given back where there is no room for them, and a failed allocation
leaves a context that can be used again.

A child process runs the library with its cudaMalloc calls under a limit (tests/alloc_limit.c, preloaded), so that
no memory of the GPU is really exhausted.
"""

import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

from gpu_util import require_gpu, to_dev, to_np, rel_l2, rand_eo

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
DIMS = (6, 4, 4, 6)
NOMEM = 3


def run(shim, limit=0, fail_at=0, scale=1.0, refused=None):
    """The results of one user's calls, and the most bytes held.  refused: a list of the calls that got
    QCD_ERR_NOMEM, each of which is then made again without a limit (None: none may)."""
    from paper_0910_0262_gb300 import qcd as Q, synth
    U, b = synth.make_problem(DIMS, 0.2, 3, 3)
    U, b = to_dev(U * scale), to_dev(b)
    op = Q.CloverWilson(DIMS, -1.0)
    shim.alloc_limit(limit, fail_at)

    def call(name, f):
        try:
            return f()
        except Q.QCDError as e:
            if refused is None or e.status != NOMEM:
                raise
            refused.append(name)
            shim.alloc_limit(0, 0)
            return f()

    call("load", lambda: op.load_gauge(U))
    call("clover", lambda: op.clover_build(0.12, 1.0))
    out = [call("op", lambda: op.dslash(b, 3, precision=64)), call("op16", lambda: op.dslash(b, 3, precision=16))]
    for prec in (32, 64):
        x, _, ok = call("solve", lambda: op.cg_solve(b, tol=1e-10, inner_prec=prec))
        assert ok
        out.append(x)
    out += [call("prepare", lambda: op.prepare_source(b, b)), call("odd", lambda: op.reconstruct_odd(b, b)),
            call("force", lambda: op.fermion_force(b, input_is_solution=True, clover_det=True)[0]),
            call("gauge", lambda: op.gauge_force(5.6))]
    out = [to_np(t) for t in out]
    peak, count = shim.alloc_peak(), shim.alloc_count()
    op.close()
    return out, peak, count


def same(a, b):
    """The two routes' rounding: FP64 1e-14, FP16 storage 1e-3, solves to 1e-10 of conditions of order ten."""
    tol = [1e-14, 2e-3, 4e-9, 4e-9, 1e-14, 1e-14, 1e-14, 1e-14]
    return all(rel_l2(x, y) < t for x, y, t in zip(a, b, tol))


def child(path):
    shim = ctypes.CDLL(path)
    shim.alloc_limit.argtypes = [ctypes.c_size_t, ctypes.c_long]
    shim.alloc_peak.restype = ctypes.c_size_t
    shim.alloc_count.restype = ctypes.c_long
    run(shim)
    want, most, count = run(shim)
    links = int(np.prod(DIMS)) * 4
    copies = links * (9 * 16) + links // 4 * 3
    # links that are not unitary to 1e-5 take the FP64 kernels: their peak less the copies' room is what these need
    _, far, _ = run(shim, scale=1.0 + 1e-3)
    need = far - copies
    assert most > need + copies, (most, far, copies)
    for limit in (need, need + 4096, (need + most) // 2, most - copies, most - 1, most):
        got, peak, _ = run(shim, limit=limit)
        assert peak <= limit and same(got, want), limit
    for k in range(1, count + 1):  # each allocation fails once
        refused = []
        got, _, _ = run(shim, fail_at=k, refused=refused)
        assert len(refused) <= 1 and same(got, want), (k, refused)
    print("ok", most, need, count)


def test_calls_that_fit_without_the_copies_are_not_refused(tmp_path):
    """Under every limit from what the FP64 kernels alone need, all calls run and agree; with any one allocation
    failing, at most that call is refused, and made again it gives the same."""
    require_gpu()
    lib = str(tmp_path / "alloc_limit.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", os.path.join(HERE, "alloc_limit.c"), "-o", lib, "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=lib)
    r = subprocess.run([sys.executable, os.path.abspath(__file__), lib], env=env, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stderr[-4000:]
    assert r.stdout.startswith("ok")


if __name__ == "__main__":
    sys.path.insert(0, os.path.dirname(HERE))
    child(sys.argv[1])
