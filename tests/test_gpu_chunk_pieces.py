"""Iterations whose chunks are of very different lengths: the long chunk's work items are cut into pieces although there are more
items than SMs, the short ones stay whole; against the oracle run chunk by chunk."""
import numpy as np
import pytest

from paper_2609_07883_b200 import workloads as W
from tests import gpu_util as G
from tests.test_gpu_multichunk import oracle_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("heads,lens,chunks", [
    ((16, 16, 64), [100, 33], [(9000, 40), (0, 1500), (0, 700)]),              # 16 items of 71 steps before 144 short ones
    ((8, 8, 128), [], [(9000, 300), (0, 1800), (0, 1100), (0, 700)]),          # two ragged groups of the long chunk
    ((16, 8, 128), [300, 17, 2000], [(12000, 65), (11000, 129), (0, 1300), (17, 900)]),  # two long chunks
])
def test_long_and_short_chunks(oracle, heads, lens, chunks, fused):
    rng = np.random.default_rng(7)
    pages = sum(-(-x // 16) for x in lens) + sum(-(-(p + c) // 16) for p, c in chunks) + 7
    batch = W.make_multi_batch(W.AttnShape(*heads), pages, lens, chunks, rng)
    t = W.host_tensors(batch, rng)
    r = G.Runner(batch, t)
    pool, out, lse = oracle_rows(oracle, batch, t)
    for _ in range(2):
        if fused:
            r.iterate()
        else:
            r.append()
            r.attend()
        got, got_lse = r.results()
        assert r.status() == (0, 0)
        assert np.array_equal(G.torch_to_bits(r.pool), pool)
        G.compare(got, got_lse, out, lse, f"{heads} {chunks}")
