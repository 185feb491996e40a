"""Calls recorded into CUDA graphs: what a replay reads has to outlive the call."""
import numpy as np
import pytest

from tests._helpers import PRF, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2209_03526_gb300")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = P.Context(0, prf_keys=PRF)
    yield c
    c.close()


@pytest.mark.parametrize("kind,bits,keys,points", [(P.KEY_DCF, 32, 8, 40001), (P.KEY_DPF, 9, 40, 30000)])
def test_evaluation_of_device_keys_replays_on_new_points(ctx, kind, bits, keys, points):
    """Keys and points on the device: a captured evaluation of all pairs reads device memory only, so
    its replays follow the points that the buffer then holds.  (Sizes that take the staged
    evaluation outside a capture: sorted and dense points.)"""
    g = np.random.default_rng(points)
    L = 28 + (24 if kind == P.KEY_DCF else 20) * bits
    draw = lambda n, top: g.integers(0, top, n, dtype=np.uint64).astype(np.uint32)  # noqa: E731
    wire = torch.zeros(keys * L, dtype=torch.uint8, device="cuda")
    ctx.keygen_device(kind, bits, to_dev(draw(keys // 2, 1 << bits)), to_dev(draw(keys // 2, 1 << 32)), bytes(16), wire)
    pts = to_dev(draw(points, 1 << 32))
    out = torch.zeros(keys * points, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=s):
        ctx.eval_device_keys(kind, bits, wire, keys, pts, out, all_pairs=True, stream=s.cuda_stream)
    want = torch.zeros_like(out)
    for _ in range(3):
        pts.copy_(to_dev(draw(points, 1 << 32)))
        ctx.eval_device_keys(kind, bits, wire, keys, pts, want, all_pairs=True)
        out.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
