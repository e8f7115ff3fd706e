"""The append where a warp takes several rows at once (rows of fewer than 32 sixteen-byte pieces) and where it takes parts of one: the
pool after it, bit for bit, with row counts that leave parts of a warp over and a row that cannot be written among good ones."""
import numpy as np
import pytest

from paper_2609_07883_b200 import workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads", [(1, 1, 64), (2, 2, 64), (8, 1, 128), (3, 3, 64), (4, 4, 64), (3, 3, 128), (6, 6, 128)])   # 8 .. 96 pieces
@pytest.mark.parametrize("lens,chunks", [
    ([17], []),
    ([5, 16, 33], [(13, 1)]),
    ([40, 1, 300, 20, 21], [(30, 67), (0, 2), (16, 18)]),
    ([100] * 7, [(5, 2500)]),
])
def test_rows_of_all_widths(oracle, heads, lens, chunks):
    rng = np.random.default_rng(41)
    shape = W.AttnShape(*heads)
    pages = sum(-(-x // 16) for x in lens) + sum(-(-(p + c) // 16) for p, c in chunks) + 4
    if len(chunks) > 1:
        batch = W.make_multi_batch(shape, pages, lens, chunks, rng)
    else:
        batch = W.make_batch(shape, pages, lens, *(chunks[0] if chunks else (0, 0)), rng)
    t = W.host_tensors(batch, rng)
    want, row = t["pool"].copy(), 0
    empty = np.zeros(0, np.int32)
    parts = [W.MixedBatch(shape, pages, P, C, ids, empty, np.zeros(1, np.int32), empty) for P, C, _, ids in batch.chunks()]
    parts.append(W.MixedBatch(shape, pages, 0, 0, empty, batch.decode_kv_len, batch.decode_page_indptr, batch.decode_pages))
    for p in parts:
        n = p.num_rows
        assert oracle.kv_append(want, p, t["k_new"][row:row + n], t["v_new"][row:row + n]) == 0
        row += n
    for fused in (False, True):
        r = G.Runner(batch, t)
        r.iterate() if fused else r.append()
        assert r.status() == (0, 0)
        assert np.array_equal(G.torch_to_bits(r.pool), want)


@pytest.mark.parametrize("heads", [(1, 1, 64), (8, 2, 64), (8, 1, 128), (4, 4, 128)])
def test_a_row_that_cannot_be_written_leaves_its_neighbours_alone(oracle, heads):
    rng = np.random.default_rng(43)
    shape = W.AttnShape(*heads)
    lens = [20, 30, 40, 50, 60, 70]
    batch = W.make_batch(shape, 40, lens, 3, 45, rng)
    t = W.host_tensors(batch, rng)
    bad = W.MixedBatch(**{**batch.__dict__})
    bad.decode_pages = batch.decode_pages.copy()
    bad.decode_pages[batch.decode_page_indptr[3] - 1] = batch.num_pages        # request 2's last page
    bad.prefill_pages = batch.prefill_pages.copy()
    bad.prefill_pages[1] = -5                                                   # positions 16 .. 31 of the chunk's prompt
    want, untouched = t["pool"].copy(), t["pool"].reshape(-1, shape.page_elems)
    assert oracle.kv_append(want, batch, t["k_new"], t["v_new"]) == 0
    for page in (batch.prefill_pages[1], batch.decode_pages[batch.decode_page_indptr[3] - 1]):
        want.reshape(-1, shape.page_elems)[page] = untouched[page]
    r = G.Runner(bad, t)
    r.append()
    assert r.status()[0] == r.B.SW_ERR_OUT_OF_RANGE
    assert np.array_equal(G.torch_to_bits(r.pool), want)
