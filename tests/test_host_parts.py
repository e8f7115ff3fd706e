"""Which host-buffer iterations are taken apart, and into parts of how many chunk rows (host arithmetic, no GPU)."""
import ctypes as C

import numpy as np
import pytest

from paper_2609_07883_b200 import binding as B
from paper_2609_07883_b200 import workloads as W
from tests.test_gpu_host_parts import PARTS, two_chunks_of_one_prompt

SMS = 148


def part_rows(batch, sms=SMS):
    struct, keep = B.host_batch_struct(batch)
    layout = B.make_layout(batch.shape, batch.num_pages)
    return B._lib.sw_host_part_rows_of(C.byref(layout), sms, C.byref(struct))


def batch_of(heads, lens, chunks):
    shape, rng = W.AttnShape(*heads), np.random.default_rng(6)
    pages = sum(-(-x // 16) for x in lens) + sum(-(-(p + c) // 16) for p, c in chunks) + 9
    if len(chunks) > 1:
        return W.make_multi_batch(shape, pages, lens, chunks, rng)
    return W.make_batch(shape, pages, lens, *(chunks[0] if chunks else (0, 0)), rng)


@pytest.mark.parametrize("heads,lens,chunks,rows", PARTS)
def test_the_iterations_of_the_gpu_tests_are_taken_apart(heads, lens, chunks, rows):
    assert part_rows(batch_of(heads, lens, chunks)) == rows < sum(c for _, c in chunks)


@pytest.mark.parametrize("heads,lens,chunks,rows", [
    ((32, 8, 128), [100] * 400, [], 0),                    # no chunk
    ((32, 8, 128), [], [(0, 341)], 0),                     # 341 rows of 12 KB are below 4 MB
    ((32, 8, 128), [], [(0, 342)], 192),
    ((32, 8, 128), [100], [(0, 341)], 192),                # the decode rows count
    # a row is 12288 bytes and 16384 flop per attended key: as long as its 267 ns on the way up at 19566 keys
    ((32, 8, 128), [], [(18989, 1152)], 576),              # more bytes than arithmetic: halves
    ((32, 8, 128), [], [(20000, 1152)], 0),                # more arithmetic than bytes: parts of 18 groups of 64 rows
    ((32, 8, 128), [], [(20000, 1153)], 1152),
    ((32, 8, 128), [60000] * 16, [(20000, 1153)], 1152),   # whatever the decode requests hold
])
def test_the_rule(heads, lens, chunks, rows):
    assert part_rows(batch_of(heads, lens, chunks)) == rows


def test_chunks_of_their_own_are_taken_apart():
    batch = W.make_multi_batch(W.LLAMA, 200, [300, 40], [(100, 500), (96, 4)], np.random.default_rng(4))
    assert part_rows(batch) == 256


def test_chunks_that_share_a_page_stay_together():
    assert part_rows(two_chunks_of_one_prompt(np.random.default_rng(4))) == 0


@pytest.mark.parametrize("page_of_chunk,together", [(31, False), (32, True), (50, True), (63, True)])
def test_a_decode_request_that_ends_on_a_page_of_the_chunk_stays_with_it(page_of_chunk, together):
    batch = W.make_batch(W.LLAMA, 200, [100], 512, 500, np.random.default_rng(3))   # rows on pages 32 .. 63 of the prompt
    batch.decode_pages = batch.prefill_pages[page_of_chunk - 6:page_of_chunk + 1].copy()
    assert (part_rows(batch) == 0) == together
