"""Decode contexts around the edges of the split and of the merge: numbers of units that fill, miss and exceed a batch of the merge.
Decode-only launches with up to 432 requests and 512 elements per group share their pages out as a line instead of units (see
test_gpu_decode_line.py): units are what the others have, and all launches with a chunk."""
import numpy as np
import pytest

from paper_2609_07883_b200 import workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def run(oracle, heads, lens, what, fused=True, chunk=0):
    rng = np.random.default_rng(51)
    shape = W.AttnShape(*heads)
    batch = W.make_batch(shape, sum(-(-x // 16) for x in lens) + 3, lens, 0, chunk, rng)
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


@pytest.mark.parametrize("heads,chunk", [((4, 4, 64), 1), ((2, 2, 128), 1), ((4, 2, 64), 1), ((8, 2, 128), 1), ((8, 1, 64), 1),
                                         ((8, 1, 128), 0), ((16, 2, 128), 0)])
def test_numbers_of_splits_of_units(oracle, heads, chunk):
    """The same numbers where the launch has units: beside a chunk of one token, and with groups of eight at head size 128."""
    for splits in (2, 7, 8, 9, 15, 16, 17, 31, 32, 33):
        run(oracle, heads, [64 * splits - 3], f"{heads}, {splits} splits, chunk {chunk}", chunk=chunk)


@pytest.mark.parametrize("fused", [True, False])
@pytest.mark.parametrize("heads", [(8, 2, 128), (4, 4, 64), (16, 4, 128)])
def test_more_requests_than_the_line_takes(oracle, heads, fused):
    """433 requests, one of them cut into many units: merges by the last ticket (one query head per KV head) and shared ones."""
    lens = [int(x) for x in np.random.default_rng(53).integers(1, 120, 433)]
    lens[200] = 20000
    run(oracle, heads, lens, f"{heads}", fused)


@pytest.mark.parametrize("heads", [(8, 2, 128), (4, 4, 64)])
def test_long_request_beside_a_one_token_chunk(oracle, heads):
    run(oracle, heads, [20000, 50], f"{heads}", chunk=1)


@pytest.mark.parametrize("heads,lens", [
    ((8, 2, 64), [128] * 9), ((8, 2, 64), [128] * 8 + [129]),                      # eight pages a context, and one more
    ((8, 1, 128), [128] * 4), ((8, 1, 128), [128] * 5), ((8, 1, 128), [112] * 4),  # four contexts or fewer
    ((8, 1, 64), [511 * 16]), ((8, 1, 64), [511 * 16 + 1]), ((8, 1, 64), [20, 512 * 16 + 5, 3]),   # 128 units of four pages and more
    ((4, 4, 64), [64]), ((4, 4, 64), [65]), ((4, 4, 64), [1, 1, 300]),
])
@pytest.mark.parametrize("chunk", [0, 1])
def test_contexts_at_the_edges_of_the_small_batch_rule(oracle, heads, lens, chunk):
    run(oracle, heads, lens, f"{heads} {len(lens)} x {max(lens)}, chunk {chunk}", chunk=chunk)


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


@pytest.mark.parametrize("heads,lens,P,C", [
    ((32, 8, 128), [int(x) for x in np.linspace(256, 2048, 64)], 512, 512),     # half of the CTAs have entries
    ((32, 8, 128), [2500] * 40, 0, 300),                                        # fewer of them
    ((32, 8, 128), [1, 16, 17, 300], 4000, 64),                                 # few units
    ((16, 4, 64), [int(x) for x in np.linspace(1, 4000, 50)], 37, 1000),
    ((16, 8, 128), [900] * 30, 100, 260),
])
@pytest.mark.parametrize("fused", [True, False])
def test_beside_a_chunk(oracle, heads, lens, P, C, fused):
    """CTAs with chunk-prefill entries come late to the decode units, which are then planned in one size or two."""
    rng = np.random.default_rng(8)
    shape = W.AttnShape(*heads)
    batch = W.make_batch(shape, sum(-(-x // 16) for x in lens) + -(-(P + C) // 16) + 3, lens, P, C, rng)
    rows = G.boundary_rows(C, heads[0] // heads[1])[::7] + list(range(C, C + len(lens)))
    pairs = [(r, int(rng.integers(heads[0]))) for r in rows]
    for seed in (73, 74):
        G.run_device_case(oracle, batch, pairs, seed, f"{heads} {len(lens)} beside {P}+{C}", fused=fused)
