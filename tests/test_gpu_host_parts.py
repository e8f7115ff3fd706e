"""Host-buffer iterations large enough to be copied and computed in parts: the parts' edges, ragged ends, several chunks, a page that
chunk rows share with a decode request, pinned and pageable buffers; against the oracle."""
import numpy as np
import pytest

from paper_2609_07883_b200 import workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def run_host(oracle, batch, pinned, with_lse, seed, rng):
    import torch

    from paper_2609_07883_b200 import binding as B

    dev = torch.device("cuda", 0)
    sh, R = batch.shape, batch.num_rows
    pages = int(batch.prefill_pages.shape[0] + batch.decode_pages.shape[0])
    ctx = B.Context(sh, batch.num_pages, batch.chunk_len, max(batch.num_decode, 1), pages + 16)
    pool = torch.empty(batch.num_pages * sh.page_elems, dtype=torch.bfloat16, device=dev)
    W.fill_normal_bf16_(pool, seed)
    gen = torch.Generator()
    gen.manual_seed(seed + 1)
    q, k, v = (torch.randn(R, h, sh.head_dim, generator=gen).to(torch.bfloat16)
               for h in (sh.num_q_heads, sh.num_kv_heads, sh.num_kv_heads))
    out = torch.zeros_like(q)
    lse = torch.zeros(R, sh.num_q_heads)
    if pinned:
        q, k, v, out, lse = (t.pin_memory() for t in (q, k, v, out, lse))
    hs, keep = B.host_batch_struct(batch)
    before = G.torch_to_bits(pool)
    results = []
    for _ in range(2):    # the first pass finds other rows in the pool; again on the same context: events and streams are kept
        out.zero_()
        B.sw_mixed_iteration_host(ctx, pool, hs, q, k, v, out, lse if with_lse else None)
        assert B.sw_check_status(ctx, raise_on_error=False) == (0, 0)
        results.append((W.bf16_bits_to_f64(G.torch_to_bits(out)), lse.numpy().astype(np.float64)))
    want = before.copy()
    rows = 0
    if batch.chunk_lens is None:
        assert oracle.kv_append(want, batch, G.torch_to_bits(k), G.torch_to_bits(v)) == 0
    else:                 # the chunks one by one, then the decodes
        for j, (P, C) in enumerate(zip(batch.chunk_prefix_lens, batch.chunk_lens)):
            one = W.MixedBatch(sh, batch.num_pages, int(P), int(C),
                               batch.prefill_pages[batch.chunk_page_indptr[j]:batch.chunk_page_indptr[j + 1]],
                               np.zeros(0, np.int32), np.zeros(1, np.int32), np.zeros(0, np.int32))
            assert oracle.kv_append(want, one, G.torch_to_bits(k[rows:rows + C]), G.torch_to_bits(v[rows:rows + C])) == 0
            rows += int(C)
        dec = W.MixedBatch(sh, batch.num_pages, 0, 0, np.zeros(0, np.int32), batch.decode_kv_len, batch.decode_page_indptr,
                           batch.decode_pages)
        assert oracle.kv_append(want, dec, G.torch_to_bits(k[rows:]), G.torch_to_bits(v[rows:])) == 0
    assert np.array_equal(G.torch_to_bits(pool), want)
    # chunk by chunk (the oracle takes one), rows around the parts' edges and a few others, one head each
    edges = {r + d for r in range(0, batch.chunk_len, 64) for d in (-1, 0)} | set(range(batch.chunk_len, R))
    at = 0
    chunks = [(batch.prefix_len, batch.chunk_len, batch.prefill_pages)] if batch.chunk_lens is None else \
        [(int(P), int(C), batch.prefill_pages[batch.chunk_page_indptr[j]:batch.chunk_page_indptr[j + 1]])
         for j, (P, C) in enumerate(zip(batch.chunk_prefix_lens, batch.chunk_lens))]
    for j, (P, C, pf) in enumerate(chunks):
        last = j == len(chunks) - 1
        n = batch.num_decode if last else 0
        one = W.MixedBatch(sh, batch.num_pages, P, C, pf, batch.decode_kv_len[:n], batch.decode_page_indptr[:n + 1], batch.decode_pages)
        take = sorted(r - at for r in edges if at <= r < at + C + n) + [0, C - 1]
        pairs = np.array([(r, int(rng.integers(sh.num_q_heads))) for r in take], dtype=np.int32)
        ref, ref_lse, _ = oracle.mixed_attention(want, one, G.torch_to_bits(q[at:at + C + n]), pairs=pairs)
        rr = pairs[:, 0] + at
        for got, got_lse in results:
            G.compare(got[rr, pairs[:, 1]], got_lse[rr, pairs[:, 1]] if with_lse else None, ref, ref_lse, f"host parts, chunk {j}")
        at += C


# (heads, decode lengths, chunks, chunk rows of a part: see test_host_parts.py)
PARTS = [
    ((32, 8, 128), [300, 17, 1, 2047], [(512, 512)], 256),            # decodes on their own
    ((32, 8, 128), [], [(0, 1001)], 512),                             # ragged last part, no decodes
    ((32, 8, 128), [40, 500], [(700, 260), (33, 300), (0, 65)], 320),  # parts that hold ends and beginnings of chunks
    ((16, 4, 64), [129], [(4111, 1777)], 896),
    ((8, 1, 128), [64, 65], [(100, 2100)], 1056),
    ((16, 4, 64), [700], [(20000, 2500)], 2368),                      # bound by the arithmetic: a first part of a whole grid's items
]


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("heads,lens,chunks", [case[:3] for case in PARTS])
def test_parts(oracle, heads, lens, chunks, pinned):
    rng = np.random.default_rng(len(lens) + heads[0])
    sh = W.AttnShape(*heads)
    need = sum(-(-x // 16) for x in lens) + sum(-(-(p + c) // 16) for p, c in chunks)
    if len(chunks) == 1:
        batch = W.make_batch(sh, need + 9, lens, chunks[0][0], chunks[0][1], rng)
    else:
        batch = W.make_multi_batch(sh, need + 9, lens, chunks, rng)
    run_host(oracle, batch, pinned, pinned, 91, rng)


def test_a_decode_row_on_a_page_of_the_chunk(oracle):
    """The decode request's last page is the chunk's last page: it attends chunk rows written by the same call."""
    rng = np.random.default_rng(3)
    batch = W.make_batch(W.LLAMA, 200, [100], 512, 500, rng)       # the chunk ends in slot 3 of its last page
    pages = batch.prefill_pages[-(-1012 // 16) - 7:-(-1012 // 16)]
    batch.decode_pages = pages.copy()
    batch.decode_kv_len = np.array([6 * 16 + 5], dtype=np.int32)   # its row is in slot 4 of that page
    batch.decode_page_indptr = np.array([0, 7], dtype=np.int32)
    run_host(oracle, batch, True, True, 92, rng)


def two_chunks_of_one_prompt(rng, decode_lens=(300, 40)):
    """Two chunks of one prompt whose rows meet on a page: 500 tokens at prefix 100, listed first, and the four tokens before them."""
    one = W.make_batch(W.LLAMA, 200, decode_lens, 100, 500, rng)
    n = one.prefill_pages.shape[0]
    return W.MixedBatch(**{**one.__dict__, "chunk_len": 504, "prefill_pages": np.concatenate([one.prefill_pages, one.prefill_pages[:7]]),
                           "chunk_prefix_lens": np.array([100, 96], np.int32), "chunk_lens": np.array([500, 4], np.int32),
                           "chunk_page_indptr": np.array([0, n, n + 7], np.int32)})


def test_chunks_that_share_a_page(oracle):
    """The rows of the second chunk are attended by the first one's, whichever part those are in."""
    rng = np.random.default_rng(4)
    run_host(oracle, two_chunks_of_one_prompt(rng), True, True, 93, rng)


@pytest.mark.parametrize("tokens", [40, 500])    # run whole, taken apart
def test_a_missing_page_list_is_refused(tokens):
    import torch

    from paper_2609_07883_b200 import binding as B

    batch = W.make_batch(W.LLAMA, 64, [], 0, tokens, np.random.default_rng(1))
    ctx = B.Context(W.LLAMA, 64, tokens, 1, 64)
    pool = torch.zeros(64 * W.LLAMA.page_elems, dtype=torch.bfloat16, device="cuda")
    q, k, v, out = (torch.zeros(tokens, h, 128, dtype=torch.bfloat16) for h in (32, 8, 8, 32))
    struct, keep = B.host_batch_struct(batch)
    struct.prefill_pages = None
    with pytest.raises(B.SwError) as e:
        B.sw_mixed_iteration_host(ctx, pool, struct, q, k, v, out)
    assert e.value.status == B.SW_ERR_INVALID_ARG
    struct, keep = B.host_batch_struct(batch)         # the context is usable afterwards
    B.sw_mixed_iteration_host(ctx, pool, struct, q, k, v, out)
    assert B.sw_check_status(ctx, raise_on_error=False) == (0, 0)
