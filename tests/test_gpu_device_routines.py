"""Single device routines of the library (compiled from device_probe.cu beside the library's headers).

* The operand ring of the triangular solves on operands that solve a diagonal matrix, exact in both
  precisions; and its bounded waits: a CTA whose copying warp is missing gets no operand, gives up after
  the limit, reports it, and leaves the device usable.
* A wait that gave up in one call: that call reports it, the next one on the same context does not.
* log x and 1 / x of the element routines against extended precision, over the whole range, next to 1, at the
  ends of the table's bins and binades, and on both sides of 2^-1007 and 2^1007, where log() and a division
  take over.  log x = (e log 2 + c) + l, |c| < 0.41, |l| < 2^-7: for |log x| < 1 (|e| <= 2) half an ulp of c
  (2.8e-17), of both sums (5.6e-17 each) and of log 2 (5.6e-17 x |e| / 2), and a few roundings of l (2e-18
  each): 2.1e-16 absolute; beyond, one ulp of the result more than covers the two sums and e times log 2's
  rounding (0.3 ulp), and log() has one: 2 ulp.  The reciprocal is one Newton step with one rounding in
  the residual and one at the end: 1 ulp.
* The pivots' reciprocal: in FP64 one rounding and a truncation of 2^-69 inside [2^-100, 2^100), a division
  outside; in FP32 the correctly rounded one.
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


def special(dtype):
    info = np.finfo(dtype)
    return np.array([0.0, -0.0, -1.0, -3.5, info.tiny, info.smallest_subnormal, 3 * info.smallest_subnormal, info.max,
                     np.inf, -np.inf, np.nan], dtype=dtype)


def ulps(got, want):
    """|got - want| in units in the last place of `want` (extended precision)."""
    return np.abs(got.astype(np.longdouble) - want) / np.spacing(np.abs(want).astype(got.dtype)).astype(np.longdouble)


def test_logarithm_and_reciprocal(probe):
    rng = np.random.default_rng(2)
    m = 200000
    edges = np.concatenate([1.0 + np.arange(-32, 65) / 128.0, [0.75, 1.5]])
    edges = np.outer(2.0 ** np.array([-1006, -500, -2, -1, 0, 1, 2, 500, 1005]), edges).ravel()
    ends = np.array([2.0 ** -1007, 2.0 ** 1007, 2.0 ** -1006, 2.0 ** 1006])
    x = np.concatenate([np.exp(rng.uniform(-1, 1, m)), rng.uniform(0.98, 1.02, m), np.exp(rng.uniform(-690, 690, m)),
                        edges, np.nextafter(edges, 0), np.nextafter(edges, np.inf),
                        ends, np.nextafter(ends, 0), np.nextafter(ends, np.inf)])
    log, inv = np.empty_like(x), np.empty_like(x)
    assert probe.probe_log_inv(x.size, ptr(x), ptr(log), ptr(inv)) == 0
    want = np.log(x.astype(np.longdouble))
    small = np.abs(want) < 1
    assert np.max(np.abs(log[small] - want[small])) <= 2.1e-16
    assert np.max(ulps(log[~small], want[~small])) <= 2
    assert np.max(ulps(inv, 1 / x.astype(np.longdouble))) <= 1
    assert log[x == 1.0][0] == 0.0
    x = special(np.float64)
    log, inv = np.empty_like(x), np.empty_like(x)
    assert probe.probe_log_inv(x.size, ptr(x), ptr(log), ptr(inv)) == 0
    with np.errstate(all="ignore"):
        want, winv = np.where(x > 0, np.log(x), 0.0), 1 / x
    finite = np.isfinite(want)
    assert np.array_equal(log[~finite], want[~finite])
    assert np.all(np.abs(log[finite] - want[finite]) <= 2 * np.spacing(np.abs(want[finite])))
    assert np.array_equal(inv, winv, equal_nan=True)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_reciprocal_of_a_pivot(probe, dtype):
    rng = np.random.default_rng(3)
    run = probe.probe_recip_f32 if dtype == np.float32 else probe.probe_recip_f64
    top = 120 if dtype == np.float32 else 1000
    powers = 2.0 ** np.array([-1000, -120, -101, -100, -99, -1, 0, 1, 99, 100, 101, 120, 1000])
    powers = powers[np.abs(np.log2(powers)) <= top].astype(dtype)
    wide, near = 2.0 ** rng.uniform(-top, top, 200000), 2.0 ** rng.uniform(-100, 100, 200000)
    x = np.concatenate([wide.astype(dtype), -near.astype(dtype), powers, np.nextafter(powers, dtype(0)),
                        np.nextafter(powers, dtype(np.inf)), special(dtype)])
    y = np.empty_like(x)
    assert run(x.size, ptr(x), ptr(y)) == 0
    with np.errstate(all="ignore"):
        exact = dtype(1) / x
    if dtype == np.float32:
        assert np.array_equal(y, exact, equal_nan=True)
        return
    plain = np.isfinite(exact) & np.isfinite(x) & (np.abs(exact) >= np.finfo(dtype).tiny)
    assert np.array_equal(y[~plain], exact[~plain], equal_nan=True)
    assert np.max(ulps(y[plain], 1 / x[plain].astype(np.longdouble))) <= 0.501
