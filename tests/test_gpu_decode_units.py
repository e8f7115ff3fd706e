"""Decode contexts around the edges of the split and of the merge: numbers of units that fill, miss and exceed a batch of the merge."""
import numpy as np
import pytest

from paper_2609_07883_b200 import workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def run(oracle, heads, lens, what, fused=True):
    rng = np.random.default_rng(51)
    shape = W.AttnShape(*heads)
    batch = W.make_batch(shape, sum(-(-x // 16) for x in lens) + 3, lens, 0, 0, rng)
    t = W.host_tensors(batch, rng)
    pool = t["pool"].copy()
    assert oracle.kv_append(pool, batch, t["k_new"], t["v_new"]) == 0
    ref, ref_lse, _ = oracle.mixed_attention(pool, batch, t["q"])
    r = G.Runner(batch, t)
    for _ in range(2):
        if fused:
            r.iterate()
        else:
            r.append()
            r.attend()
        assert r.status() == (0, 0)
        out, lse = r.results()
        G.compare(out.reshape(-1, shape.head_dim), lse.reshape(-1), ref, ref_lse, what)


@pytest.mark.parametrize("heads", [(4, 4, 64), (2, 2, 128), (4, 2, 64), (8, 2, 128), (8, 1, 64)])
def test_numbers_of_splits_around_a_batch_of_the_merge(oracle, heads):
    for splits in (2, 7, 8, 9, 15, 16, 17, 31, 32, 33):   # units of 64 tokens
        run(oracle, heads, [64 * splits - 3], f"{heads}, {splits} splits")


@pytest.mark.parametrize("heads,lens", [
    ((8, 2, 64), [128] * 9), ((8, 2, 64), [128] * 8 + [129]),                      # eight pages a context, and one more
    ((8, 1, 128), [128] * 4), ((8, 1, 128), [128] * 5), ((8, 1, 128), [112] * 4),  # four contexts or fewer
    ((8, 1, 64), [511 * 16]), ((8, 1, 64), [511 * 16 + 1]), ((8, 1, 64), [20, 512 * 16 + 5, 3]),   # 128 units of four pages and more
    ((4, 4, 64), [64]), ((4, 4, 64), [65]), ((4, 4, 64), [1, 1, 300]),
])
def test_contexts_at_the_edges_of_the_small_batch_rule(oracle, heads, lens):
    run(oracle, heads, lens, f"{heads} {len(lens)} x {max(lens)}")


@pytest.mark.parametrize("heads", [(8, 1, 64), (16, 2, 128), (8, 2, 64), (4, 2, 64), (8, 2, 128)])
def test_requests_of_1_to_30_units_beside_a_chunk(oracle, heads):
    """Beside chunk-prefill entries not every unit has a warp of its own: merges by the last ticket and shared ones in one launch."""
    rng = np.random.default_rng(52)
    shape = W.AttnShape(*heads)
    lens = [int(x) for x in np.linspace(20, 3900, 40)]
    for fused in (True, False):
        batch = W.make_batch(shape, sum(-(-x // 16) for x in lens) + 40, lens, 100, 400, rng)
        t = W.host_tensors(batch, rng)
        pool = t["pool"].copy()
        assert oracle.kv_append(pool, batch, t["k_new"], t["v_new"]) == 0
        ref, ref_lse, _ = oracle.mixed_attention(pool, batch, t["q"])
        r = G.Runner(batch, t)
        for _ in range(2):
            if fused:
                r.iterate()
            else:
                r.append()
                r.attend()
            assert r.status() == (0, 0)
            out, lse = r.results()
            G.compare(out.reshape(-1, shape.head_dim), lse.reshape(-1), ref, ref_lse, f"{heads} fused={fused}")
