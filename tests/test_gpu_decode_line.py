"""Decode-only launches whose stages are shared out in a line: stretches shorter than a CTA's warps, pairs on one warp, on several and on
several CTAs, the largest batch of the rule and the first one beyond it, page lists that are too short, waits that expire."""
import ctypes

import numpy as np
import pytest

from paper_2609_07883_b200 import workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def run(oracle, heads, lens, what, fused=True, seed=71):
    rng = np.random.default_rng(seed)
    shape = W.AttnShape(*heads)
    batch = W.make_batch(shape, sum(-(-x // 16) for x in lens) + 3, lens, 0, 0, rng)
    t = W.host_tensors(batch, rng)
    pool = t["pool"].copy()
    assert oracle.kv_append(pool, batch, t["k_new"], t["v_new"]) == 0
    ref, ref_lse, _ = oracle.mixed_attention(pool, batch, t["q"])
    r = G.Runner(batch, t)
    for _ in range(2):                      # the second launch finds the tickets re-armed
        if fused:
            r.iterate()
        else:
            r.append()
            r.attend()
        assert r.status() == (0, 0)
        out, lse = r.results()
        G.compare(out.reshape(-1, shape.head_dim), lse.reshape(-1), ref, ref_lse, what)
        assert np.array_equal(G.torch_to_bits(r.pool).reshape(-1), pool.reshape(-1)), what


@pytest.mark.parametrize("fused", [True, False])
@pytest.mark.parametrize("heads", [(4, 1, 128), (2, 2, 128), (8, 1, 64), (4, 4, 64), (4, 2, 64)])
def test_stretches_and_pairs(oracle, heads, fused):
    for lens in ([1], [16 * 11], [16 * 12], [16 * 13 - 1], [1] * 13, [16 * 25, 1, 17, 16 * 40 - 3],   # up to a few CTAs
                 [16 * 148 * 12], [16 * 148 * 12 + 1], [16 * 1777, 5],                                 # one page a warp of one head, and one more
                 [int(x) for x in np.linspace(1, 1500, 60)]):                                          # pairs on one warp and on several
        run(oracle, heads, lens, f"{heads} {len(lens)} x {max(lens)}", fused)


@pytest.mark.parametrize("n", [432, 433])
def test_largest_batch_of_the_line(oracle, n):
    run(oracle, (4, 1, 128), [int(x) for x in np.random.default_rng(n).integers(1, 90, n)], f"{n} requests")


@pytest.mark.parametrize("fused", [True, False])
@pytest.mark.parametrize("heads,lens", [
    ((8, 2, 128), [16 * 13 - 9] * 300),                                        # four or five pages a warp: nearly every pair is cut
    ((32, 8, 128), [int(x) for x in np.random.default_rng(6).integers(150, 330, 90)]),
    ((8, 2, 64), [16 * 17 + 1, 16 * 11 - 1] * 130),
])
def test_page_buffers_are_refilled_behind_pairs_that_end_in_a_warp(oracle, heads, lens, fused):
    """A pair that an earlier warp began ends in a partly filled page whose buffer is written with plain stores (the new row, zeroed rows)
    and then refilled with the next pair's page: no such store may land on that page.  The unwritten slots of the pool hold NaNs."""
    rng = np.random.default_rng(79)
    shape = W.AttnShape(*heads)
    batch = W.make_batch(shape, sum(-(-x // 16) for x in lens) + 3, lens, 0, 0, rng)
    t = W.host_tensors(batch, rng)
    pool = t["pool"].reshape(batch.num_pages, 2, shape.num_kv_heads, 16, shape.head_dim)
    for i, x in enumerate(lens):
        page = batch.decode_pages[batch.decode_page_indptr[i + 1] - 1]
        pool[page, :, :, (x - 1) % 16 + 1:] = 0x7FC0
    after = t["pool"].copy()
    assert oracle.kv_append(after, batch, t["k_new"], t["v_new"]) == 0
    ref, ref_lse, _ = oracle.mixed_attention(after, batch, t["q"])
    r = G.Runner(batch, t)
    first = None
    for _ in range(10):
        if fused:
            r.iterate()
        else:
            r.append()
            r.attend()
        out, lse = r.results()
        if first is None:
            assert r.status() == (0, 0)
            G.compare(out.reshape(-1, shape.head_dim), lse.reshape(-1), ref, ref_lse, f"{heads}")
            first = out, lse
        assert np.array_equal(out, first[0]) and np.array_equal(lse, first[1])


@pytest.mark.parametrize("fused", [True, False])
@pytest.mark.parametrize("heads,lens", [((32, 8, 128), [2000] * 64), ((8, 2, 64), [30000, 500] * 12), ((4, 1, 128), [200000])])
def test_expired_waits_leave_no_wrong_rows(oracle, heads, lens, fused):
    """With a limit of zero most waits for a page expire.  The launch is reported, and every row of the output is right or untouched."""
    rng = np.random.default_rng(80)
    shape = W.AttnShape(*heads)
    batch = W.make_batch(shape, sum(-(-x // 16) for x in lens) + 3, lens, 0, 0, rng)
    t = W.host_tensors(batch, rng)
    pool = t["pool"].copy()
    assert oracle.kv_append(pool, batch, t["k_new"], t["v_new"]) == 0
    ref, ref_lse, _ = oracle.mixed_attention(pool, batch, t["q"])
    r = G.Runner(batch, t)
    if not fused:
        r.append()
    launch = r.iterate if fused else r.attend
    assert r.B._lib.sw_ctx_set_line_wait(r.ctx.handle, ctypes.c_int64(0)) == r.B.SW_OK
    for _ in range(3):
        r.out.zero_()
        r.lse.zero_()
        launch()
        assert r.status()[0] == r.B.SW_ERR_DEVICE_TIMEOUT
        out, lse = (x.reshape(ref.shape[0], -1) for x in r.results())
        done = (out != 0).any(1) | (lse[:, 0] != 0)
        assert not done.all()
        if done.any():
            G.compare(out[done], lse[done, 0], ref[done], ref_lse[done], f"{heads}: {done.sum()} rows")
    assert r.B._lib.sw_ctx_set_line_wait(r.ctx.handle, ctypes.c_int64(2_000_000_000)) == r.B.SW_OK
    launch()                                # the tickets are re-armed
    assert r.status() == (0, 0)
    out, lse = r.results()
    G.compare(out.reshape(-1, shape.head_dim), lse.reshape(-1), ref, ref_lse, f"{heads} afterwards")


@pytest.mark.parametrize("fused", [True, False])
@pytest.mark.parametrize("heads", [(32, 8, 128), (8, 2, 64), (8, 1, 64), (2, 2, 128)])
def test_short_contexts_are_not_cut(oracle, heads, fused):
    """Launches whose pairs all go whole to a warp, and the first ones with a pair that is too long for that."""
    rng = np.random.default_rng(83)
    for lens in ([1], [128], [129], [128] * 5, [129] + [16] * 4, [1] * 432, [16, 17] * 100,
                 [int(x) for x in rng.integers(1, 129, 40)], [int(x) for x in rng.integers(1, 129, 432)],
                 [int(x) for x in rng.integers(100, 20 * 16 + 1, 432)],                      # more stages: up to 20 and 24 are whole
                 [24 * 16] * 432, [24 * 16] * 431 + [24 * 16 + 1], [20 * 16 + 1] * 432):
        if fused or len(lens) * max(lens) < 30000:
            run(oracle, heads, lens, f"{heads} {len(lens)} x {max(lens)}", fused)


def test_long_stretches(oracle):
    """Two pairs of 100000 and 13000 pages: 64 pages a warp and more."""
    batch = W.make_batch(W.AttnShape(1, 1, 64), 113003, [16 * 100000 - 3, 16 * 13000 - 7], 0, 0, np.random.default_rng(3))
    G.run_device_case(oracle, batch, None, 72, "long stretches", fused=True)


@pytest.mark.parametrize("heads", [(8, 8, 64), (32, 8, 128)])
def test_more_than_two_to_the_23_stages(oracle, heads):
    """Page lists that name the same pages again and again: 1.1 million pages per KV head of a pool of 4000."""
    rng = np.random.default_rng(81)
    shape = W.AttnShape(*heads)
    batch = W.make_batch(shape, 4000, [16 * 3000 - 5, 16 * 900 - 1, 33], 0, 0, rng)
    times = [240, 430, 1]                                           # the list of request i is its pages, that often, last page last
    lists = [np.tile(batch.decode_pages[a:b], k) for a, b, k in zip(batch.decode_page_indptr, batch.decode_page_indptr[1:], times)]
    for x in lists[:2]:                                             # full pages in the middle: other ones than the last
        x[:-1][x[:-1] == x[-1]] = x[0]
    pages = np.array([len(x) for x in lists])
    batch.decode_kv_len = (16 * pages - np.array([5, 1, 15])).astype(np.int32)
    batch.decode_page_indptr = np.concatenate([[0], np.cumsum(pages)]).astype(np.int32)
    batch.decode_pages = np.concatenate(lists).astype(np.int32)
    assert pages.sum() * shape.num_kv_heads > 1 << 23
    pairs = [(0, 0), (0, heads[0] - 1), (1, heads[0] // 2), (2, 1)]
    G.run_device_case(oracle, batch, pairs, 82, f"{heads}, {pages.sum()} pages", fused=True)


@pytest.mark.parametrize("fused", [True, False])
def test_requests_with_short_page_lists(oracle, fused):
    """Requests whose list ends before their context are reported and get no output (and no new row); the others' are right."""
    rng = np.random.default_rng(5)
    shape = W.AttnShape(8, 2, 128)
    lens = [700, 16 * 30, 4000, 33, 9]
    batch = W.make_batch(shape, sum(-(-x // 16) for x in lens) + 3, lens, 0, 0, rng)
    t = W.host_tensors(batch, rng)
    pool = t["pool"].copy()
    if fused:
        assert oracle.kv_append(pool, batch, t["k_new"], t["v_new"]) == 0
    ref, ref_lse, _ = oracle.mixed_attention(pool, batch, t["q"])
    batch.decode_kv_len = batch.decode_kv_len.copy()
    batch.decode_kv_len[[1, 3]] += 16
    r = G.Runner(batch, t)
    if fused:
        r.iterate()
        per_page = t["pool"].size // batch.num_pages
        for i in (1, 3):                                            # their pages hold what they held
            ids = batch.decode_pages[batch.decode_page_indptr[i]:batch.decode_page_indptr[i + 1]]
            pool.reshape(-1, per_page)[ids] = t["pool"].reshape(-1, per_page)[ids]
        assert np.array_equal(G.torch_to_bits(r.pool).reshape(-1), pool.reshape(-1))
    else:
        r.attend()
    assert r.status()[0] == r.B.SW_ERR_OUT_OF_RANGE
    out, lse = r.results()
    good = [0, 2, 4]
    ref, ref_lse = ref.reshape(5, 8, 128), ref_lse.reshape(5, 8)
    G.compare(out[good].reshape(-1, 128), lse[good].reshape(-1), ref[good].reshape(-1, 128), ref_lse[good].reshape(-1), "good requests")
    assert not out[[1, 3]].any() and not lse[[1, 3]].any()
