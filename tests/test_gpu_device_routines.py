"""Single device routines of the library (compiled from device_probe.cu beside the library's headers).

* The operand ring of the triangular solves on operands that solve a diagonal matrix, exact in both
  precisions; and its bounded waits: a CTA whose copying warp is missing gets no operand, gives up after
  the limit, reports it, and leaves the device usable.
* A wait that gave up in one call: that call reports it, the next one on the same context does not.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2410_24138_gb300 import build
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device_probe.cu")
    lib = str(tmp_path_factory.mktemp("probe") / "libprobe.so")
    subprocess.run([build.NVCC, build.GENCODE, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
                    "-shared", "-I", build.INCLUDE, "-I", build.CSRC, src, "-o", lib], check=True)
    return ctypes.CDLL(lib)


def ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


def diagonal_operands(dtype, n, b, scale):
    """Packed operands of a matrix with inv(L) = 1 and inv(U) = scale: rows of BS entries, entry j of row r
    at ((j / G) ^ (r mod 8)) G + j mod G."""
    BS, G = (32, 4) if dtype == np.float32 else (16, 2)
    nblk = (n + BS - 1) // BS
    P = np.zeros((nblk, 2 * BS * BS + 2 * b * BS), dtype=dtype)
    for r in range(BS):
        at = r * BS + ((r // G) ^ (r & 7)) * G + r % G
        P[:, at] = 1
        P[:, BS * BS + at] = scale
    return P


@pytest.mark.parametrize("n,b,stages", [(1, 0, 2), (33, 1, 2), (200, 40, 2), (1000, 83, 3), (3000, 112, 6)])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_ring(probe, n, b, stages, dtype):
    run = probe.probe_ring_f32 if dtype == np.float32 else probe.probe_ring_f64
    P = diagonal_operands(dtype, n, b, 0.25)
    ok = ctypes.c_int(-1)
    x = np.arange(1, n + 1).astype(dtype)
    assert run(n, b, ptr(P), ptr(x), stages, 0, ctypes.byref(ok)) == 0
    assert ok.value == 1 and np.array_equal(x, 0.25 * np.arange(1, n + 1).astype(dtype))
    if n > 200:
        return
    assert run(n, b, ptr(P), ptr(x.copy()), stages, 1, ctypes.byref(ok)) == 0
    assert ok.value == 0
    assert run(n, b, ptr(P), ptr(x), stages, 0, ctypes.byref(ok)) == 0
    assert ok.value == 1 and np.array_equal(x, 0.0625 * np.arange(1, n + 1).astype(dtype))


@pytest.mark.parametrize("factor", ["band", "tiles"])
@pytest.mark.parametrize("call", ["solve", "eval_Fx", "apply_tangent"])
def test_report_of_a_wait_ends_with_its_call(probe, call, factor):
    from paper_2410_24138_gb300 import inputs as I, nls
    p = I.diffusion_problem(24, I.box_partition(24, 4, 4), 16, 1)
    s = nls.make_solver(p, coupling="hybrid", coarse_factor=getattr(nls, "COARSE_FACTOR_" + factor.upper()),
                        coarse_reuse=0)  # a call then depends on its inputs alone
    rng = np.random.default_rng(0)
    u = 0.05 * rng.random(p.n_nodes)
    u[p.dirichlet_nodes] = 0.0
    s.eval_Fx(u)

    def run():
        out = getattr(s, call)(u.copy())
        return out[0] if isinstance(out, tuple) else out

    want = run()
    tiles = probe.probe_report_wait(s.h)
    assert tiles == (factor == "tiles")
    with pytest.raises(nls.NLSError) as err:
        run()
    assert err.value.status == -9
    s.eval_Fx(u)
    assert np.array_equal(run(), want)
