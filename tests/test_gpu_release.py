"""What oblivgm_release does with a served result's memory: it goes back in order after the reads
that the caller has queued, or it stays reserved."""
import ctypes

import numpy as np
import pytest

import oracle
import workload as W
from tests._helpers import PRF, load_tables

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2209_03526_gb300")

N = 5003
BYTES = 3 * 4 * N


def _cudart():
    """the runtime that torch has loaded, for a stream that synchronises with the default stream"""
    with open("/proc/self/maps") as f:
        paths = sorted({line.split()[-1] for line in f if "libcudart.so" in line})
    lib = ctypes.CDLL(paths[0] if paths else "libcudart.so")
    lib.cudaStreamCreate.argtypes = [ctypes.POINTER(ctypes.c_void_p)]
    lib.cudaStreamBeginCapture.argtypes = [ctypes.c_void_p, ctypes.c_int]
    lib.cudaStreamEndCapture.argtypes = [ctypes.c_void_p, ctypes.POINTER(ctypes.c_void_p)]
    lib.cudaGraphDestroy.argtypes = [ctypes.c_void_p]
    lib.cudaStreamDestroy.argtypes = [ctypes.c_void_p]
    return lib


@pytest.fixture()
def served():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = W.rng(4)
    wl = {"tables": [W.table(W.uniform_attrs(g, 1, N, 16), 16, g)]}
    v = wl["tables"][0]["values"]
    preds = [[W.eq_pred(0, 0, 0, int(v[0, k]))] for k in range(2)]
    with P.Context(0, prf_keys=PRF, serve_arena_bytes=BYTES + 100) as c:
        load_tables(c, wl)
        yield c, v, preds, [P.keygen(p, 16, bytes([k]) * 16) for k, p in enumerate(preds)]


def test_a_capture_of_the_default_stream_s_kind_defers_the_free(served):
    """While a stream that synchronises with the default stream captures, no event can be recorded
    there: the memory stays reserved, a submit that needs it is refused, and once the capture
    has ended the next submit frees it."""
    ctx, v, preds, toks = served
    rt = _cudart()
    first = ctx.submit(toks[0])
    ctx.poll(first, -1)
    torch.cuda.synchronize()
    s, graph = ctypes.c_void_p(), ctypes.c_void_p()
    assert rt.cudaStreamCreate(ctypes.byref(s)) == 0
    try:
        assert rt.cudaStreamBeginCapture(s, 2) == 0          # relaxed
        try:
            ctx.release(first)
            assert ctx.serve_stats()["reserved_bytes"] == BYTES
            with pytest.raises(P.OblivgmError) as e:
                ctx.submit(toks[1])
            assert e.value.status == P.EAGAIN
        finally:
            status = rt.cudaStreamEndCapture(s, ctypes.byref(graph))
            if graph.value:
                rt.cudaGraphDestroy(graph)
        assert status == 0                                    # the release left the capture alone
    finally:
        rt.cudaStreamDestroy(s)
    second = ctx.submit(toks[1])
    assert ctx.serve_stats()["reserved_bytes"] == BYTES
    ctx.poll(second, -1)
    ctx.release(second)
    assert ctx.serve_stats()["reserved_bytes"] == 0


def test_reads_queued_on_the_default_stream_see_their_result(served):
    """A copy queued behind a long kernel on the default stream, the release at once, and the next query
    into the same memory: the copy is the first query's result."""
    ctx, v, preds, toks = served
    busy = torch.randn(4096, 4096, device="cuda")
    for rep in range(4):
        k = rep % 2
        t = ctx.submit(toks[k])
        res = ctx.poll(t, -1)
        for _ in range(20):
            busy = torch.nn.functional.normalize(busy @ busy)
        copies = [P.device_words(x, N).clone() for x in res["groups"][0]["shares"]]
        ctx.release(t)
        other = ctx.submit(toks[1 - k])
        ctx.poll(other, -1)
        ctx.release(other)
        torch.cuda.synchronize()
        rec = oracle.reconstruct(np.stack([c.cpu().numpy().view(np.uint32) for c in copies]))
        assert np.array_equal(rec, oracle.plain_group(preds[k], 0, v)), rep
