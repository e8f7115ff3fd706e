"""Fused decode-only launches write a request's new K/V row from the units that reach its last page; requests that share that page
must see each other's rows."""
import numpy as np
import pytest

from paper_2609_07883_b200 import workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def drafts(shape, sequences, others, rng):
    """A batch in which every (cached, n) of `sequences` stands for n requests of cached + 1 .. cached + n tokens over the same
    pages (tokens of one sequence verified side by side), mixed with ordinary requests of `others` tokens."""
    base = W.make_batch(shape, sum(-(-(c + n) // 16) for c, n in sequences) + sum(-(-x // 16) for x in others) + 5,
                        [c + n for c, n in sequences] + list(others), 0, 0, rng)
    reqs = []
    for i, (cached, n) in enumerate(sequences):
        pages = base.decode_pages[base.decode_page_indptr[i]:base.decode_page_indptr[i + 1]]
        reqs += [(cached + k + 1, pages[:-(-(cached + k + 1) // 16)]) for k in range(n)]
    for i, x in enumerate(others, start=len(sequences)):
        reqs.append((x, base.decode_pages[base.decode_page_indptr[i]:base.decode_page_indptr[i + 1]]))
    reqs = [reqs[i] for i in rng.permutation(len(reqs))]
    base.decode_kv_len = np.array([x for x, _ in reqs], dtype=np.int32)
    base.decode_page_indptr = np.concatenate([[0], np.cumsum([len(p) for _, p in reqs])]).astype(np.int32)
    base.decode_pages = np.concatenate([p for _, p in reqs]).astype(np.int32)
    return base


@pytest.mark.parametrize("heads", [(32, 8, 128), (16, 4, 64), (8, 1, 128), (4, 4, 64)])
@pytest.mark.parametrize("sequences,others", [
    ([(0, 16)], []),                                             # a whole page of drafts, the first token among them
    ([(100, 4), (16, 3), (95, 1)], [1, 16, 17, 4000]),           # first slots, last slots, a page of its own
    ([(5000, 5), (160, 8)], [int(x) for x in range(30, 90)]),    # more than 32 requests; one page shared by many units
])
def test_requests_that_share_their_last_page(oracle, heads, sequences, others):
    rng = np.random.default_rng(len(others) + heads[0])
    batch = drafts(W.AttnShape(*heads), sequences, others, rng)
    for _ in range(2):
        G.run_device_case(oracle, batch, None, 11, f"drafts {heads}", fused=True)


def test_a_bad_last_page_is_reported_and_nothing_is_written(oracle):
    rng = np.random.default_rng(5)
    batch = W.make_batch(W.TINY, 64, [40, 70, 33], 0, 0, rng)
    t = W.host_tensors(batch, rng)
    for bad_id in (-1, batch.num_pages, -(1 << 31)):
        bad = W.MixedBatch(**{**batch.__dict__})
        bad.decode_pages = batch.decode_pages.copy()
        bad.decode_pages[bad.decode_page_indptr[2] - 1] = bad_id
        r = G.Runner(bad, t)
        r.iterate()
        assert r.status()[0] == r.B.SW_ERR_OUT_OF_RANGE
        want = t["pool"].copy()
        keep = W.make_batch(W.TINY, 64, [40, 33], 0, 0, np.random.default_rng(5))
        keep.decode_page_indptr = np.array([0, 3, 6], dtype=np.int32)
        keep.decode_pages = np.concatenate([batch.decode_pages[:3], batch.decode_pages[batch.decode_page_indptr[2]:]])
        assert oracle.kv_append(want, keep, t["k_new"][[0, 2]], t["v_new"][[0, 2]]) == 0
        assert np.array_equal(G.torch_to_bits(r.pool), want)   # the good requests' rows and nothing else
        r.dbatch = r.B.DeviceBatch(batch, r.dev)               # the context is usable afterwards
        r.iterate()
        assert r.status() == (0, 0)


@pytest.mark.parametrize("heads", [(32, 8, 128), (16, 4, 64), (4, 4, 64)])
@pytest.mark.parametrize("empty_len", [0, -1, -14, -(1 << 31)])
def test_bad_last_pages_beside_requests_without_a_row(oracle, heads, empty_len):
    """Requests whose last page lies outside the pool and requests of length 0 or less in one batch, in either order: both are
    reported, and every other request's output and row are what they are without them."""
    shape = W.AttnShape(*heads)
    rng = np.random.default_rng(23)
    lens = [40, 33, 7, 300, 16, 95, 1, 20, 50]
    base = W.make_batch(shape, sum(-(-x // 16) for x in lens) + 3, lens, 0, 0, rng)
    t = W.host_tensors(base, rng)
    broken_page, broken_len = (0, 4, 7), (1, 3, 8)
    bad = W.MixedBatch(**{**base.__dict__})
    bad.decode_pages = base.decode_pages.copy()
    bad.decode_kv_len = base.decode_kv_len.copy()
    for i in broken_page:
        bad.decode_pages[bad.decode_page_indptr[i] + (lens[i] - 1) // 16] = -1 if i else bad.num_pages
    for i in broken_len:
        bad.decode_kv_len[i] = empty_len
    good = [i for i in range(len(lens)) if i not in broken_page + broken_len]
    keep = W.MixedBatch(**{**base.__dict__})
    keep.decode_kv_len = base.decode_kv_len[good]
    keep.decode_pages = np.concatenate([base.decode_pages[base.decode_page_indptr[i]:base.decode_page_indptr[i + 1]] for i in good])
    keep.decode_page_indptr = np.concatenate([[0], np.cumsum([-(-lens[i] // 16) for i in good])]).astype(np.int32)
    pool = t["pool"].copy()
    assert oracle.kv_append(pool, keep, t["k_new"][good], t["v_new"][good]) == 0
    ref, ref_lse, _ = oracle.mixed_attention(pool, keep, t["q"][good])
    r = G.Runner(bad, t)
    for _ in range(2):
        r.iterate()
        assert r.status()[0] == r.B.SW_ERR_OUT_OF_RANGE
        out, lse = r.results()
        assert np.array_equal(G.torch_to_bits(r.pool), pool)
        G.compare(out[good].reshape(-1, shape.head_dim), lse[good].reshape(-1), ref, ref_lse, f"{heads} {empty_len}")
