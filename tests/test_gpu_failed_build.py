"""Builds that fail on the host and are repeated, and builds of different modes in turn.

The failure is a build on a stream that is being captured: its work is recorded, not run, and its first
wait is an error."""
import ctypes

import numpy as np
import pytest

import oracle
import paper_2009_12505_gb300 as hfx
import synth
from gpu_common import compare_full, gpu_build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

THETA = 3e-2


@pytest.fixture(scope="module")
def workloads():
    """One atom with all its images within 3.2 (more than two words of 32 neighbours): C as drawn, and
    each block scaled so that the order of their largest values is reversed."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s = synth.custom("images", 1.0, 1, [[0, 0, 0]], 2, 3)
    a, b = (synth.make_workload(s, 3.2, 2.0, 3.0, seed=3) for _ in range(2))
    assert len(b.C.keys) > 96
    big = np.maximum.reduceat(np.abs(b.C.data), b.C.offs[:-1])
    b.C.data[:] = b.C.data * np.repeat(2.0 / big ** 2 * big.min(), np.diff(b.C.offs))
    return a, b


def _context(wl):
    stream = torch.cuda.Stream()
    ctx = hfx.Context(wl.system.nao, wl.system.nabf, stream=stream.cuda_stream)
    for k in "CVD":
        ctx.set_blocks(k, getattr(wl, k))
    return ctx, stream


def _failing_build(ctx, stream, *mode):
    cuda, graph = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p()
    st = ctypes.c_void_p(stream.cuda_stream)
    assert cuda.cuStreamBeginCapture_v2(st, 2) == 0  # relaxed mode
    try:
        with pytest.raises(hfx.HfxError):
            ctx.build(THETA, *mode)
    finally:
        cuda.cuStreamEndCapture(st, ctypes.byref(graph))


def _same_as_fresh(wl, ctx, *mode):
    got = gpu_build(wl, THETA, *mode, ctx=ctx)[1]
    _, ref = gpu_build(wl, THETA, *mode)
    assert len(ref["keys"]) > 0
    np.testing.assert_array_equal(got["keys"], ref["keys"])
    assert list(got["stats"]["survivors"]) == list(ref["stats"]["survivors"])
    np.testing.assert_array_equal(got["data"], ref["data"])
    assert got["ex"] == ref["ex"]


@pytest.mark.parametrize("mode", [("fp64", 0), ("ozaki", 6)])
def test_failure_is_reported_once(workloads, mode):
    """The repeated build does not fail on the error that the failed one returned."""
    ctx, stream = _context(workloads[0])
    ctx.build(THETA, *mode)
    _failing_build(ctx, stream, *mode)
    _same_as_fresh(workloads[0], ctx, *mode)


@pytest.mark.parametrize("mode", [("fp64", 0), ("ozaki", 6)])
def test_repeat_after_new_values(workloads, mode):
    """C got new values before the failed build.  The screen ends a row at the first 32 neighbours that
    all fall, so with an order or upper limits older than the values it would lose terms."""
    a, b = workloads
    ctx, stream = _context(a)
    ctx.build(THETA, *mode)
    ctx.set_blocks("C", b.C)
    _failing_build(ctx, stream, *mode)
    _same_as_fresh(b, ctx, *mode)


@pytest.mark.parametrize("nslices", [4, 6])
def test_split_after_fp64(workloads, nslices):
    """C got new values and an FP64 build before the split build of the same digit count."""
    a, b = workloads
    ctx, _ = _context(a)
    ctx.build(THETA, "ozaki", nslices)
    ctx.set_blocks("C", b.C)
    ctx.build(THETA, "fp64")
    _same_as_fresh(b, ctx, "ozaki", nslices)


@pytest.mark.parametrize("mode,tol", [(("fp64", 0), 1e-10), (("ozaki", 6), 1e-8)])
def test_new_order_matches_oracle(workloads, mode, tol):
    """C in the reverse order of size, set into a context that was built with the old order."""
    a, b = workloads
    ctx, _ = _context(a)
    ctx.build(THETA, *mode)
    ctx.set_blocks("C", b.C)
    compare_full(b, THETA, gpu_build(b, THETA, *mode, ctx=ctx)[1], oracle.Oracle.of(b).build(THETA), tol)
