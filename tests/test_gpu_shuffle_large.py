"""secShuffle (Alg. 5) on both sides of the row count up to which its round tables are kept in
shared memory and its mask blocks start from shared prefixes (2^24 rows)."""
import numpy as np
import pytest

import oracle
import workload as W
from tests._helpers import PRF, from_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2209_03526_gb300")

SEEDS = bytes(range(100, 148))


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = P.Context(0, prf_keys=PRF)
    yield c
    c.close()


@pytest.mark.parametrize("n,w", [(1 << 24, 2), ((1 << 24) + 3, 3)])
def test_shuffle_past_the_shared_round_tables(ctx, n, w):
    """2^24 rows (the largest with the round tables in shared memory and shared mask prefixes)
    and a few more (the general path): sampled rows land where the oracle's permutations put
    them, and the output masks R1, R2 are the oracle's AES blocks of the row."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    ins = [torch.randint(-(1 << 31), 1 << 31, (n, w), dtype=torch.int32, device="cuda", generator=gen) for _ in range(3)]
    outs = [torch.zeros_like(ins[0]) for _ in range(3)]
    ctx.shuffle(ins, SEEDS, outs, group=oracle.SHUF_XOR)
    torch.cuda.synchronize()
    g = W.rng(n)
    for i in [0, n - 1, (1 << 24) - 1] + [int(v) for v in g.integers(0, n, 60)]:
        j = oracle.prp(SEEDS[0:16], n, i)
        k = oracle.prp(SEEDS[32:48], n, j)
        l = oracle.prp(SEEDS[16:32], n, k)
        d = from_dev(ins[0][i] ^ ins[1][i] ^ ins[2][i])
        assert np.array_equal(from_dev(outs[0][l] ^ outs[1][l] ^ outs[2][l]), d), i
        blk = l.to_bytes(8, "little") + (2).to_bytes(2, "little") + bytes(6)
        for out, seed in ((outs[0], SEEDS[32:48]), (outs[1], SEEDS[0:16])):
            want = np.frombuffer(oracle.aes128(seed, blk), dtype=np.uint32)[:w]
            assert np.array_equal(from_dev(out[l]), want), i
