"""Which host-buffer iterations are taken apart, and into parts of how many chunk rows (host arithmetic, no GPU)."""
import ctypes as C

import numpy as np
import pytest

from paper_2609_07883_b200 import binding as B
from paper_2609_07883_b200 import workloads as W
from tests.test_gpu_host_parts import two_chunks_of_one_prompt

SMS = 148


def part_rows(batch, sms=SMS):
    struct, keep = B.host_batch_struct(batch)
    layout = B.make_layout(batch.shape, batch.num_pages)
    return B._lib.sw_host_part_rows_of(C.byref(layout), sms, C.byref(struct))


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
