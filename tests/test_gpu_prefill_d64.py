"""Chunk prefill at head size 64, whose score products run a step ahead: entries of one, two and three steps, tiles with different numbers
of steps, chunks that fill one tile only, pieces of items."""
import numpy as np
import pytest

from paper_2609_07883_b200 import workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads", [(2, 2, 64), (4, 2, 64), (4, 1, 64), (8, 1, 64)])
@pytest.mark.parametrize("P,C", [(0, 1), (0, 33), (100, 28), (0, 129), (0, 300), (127, 1), (128, 130), (255, 257), (700, 90), (3000, 200)])
def test_few_steps(oracle, heads, P, C):
    batch = W.make_batch(W.AttnShape(*heads), -(-(P + C) // 16) + 3, [], P, C, np.random.default_rng(P + C))
    for fused in (True, False):
        G.run_device_case(oracle, batch, None, 81, f"{heads} {P}+{C} fused={fused}", fused=fused)


def test_growing_scores(oracle):
    """Every step's keys raise the row maxima by more than 2^8, so that O is rescaled in every one."""
    batch = W.make_batch(W.AttnShape(4, 1, 64), 80, [], 700, 400, np.random.default_rng(9))

    def patch(pool, q, k_new, v_new):
        q[..., 0] = 8
        for i, page in enumerate(batch.prefill_pages[:700 // 16]):
            pool[int(page), 0, :, :, 0] = float(i // 8 * 20)

    G.run_device_case(oracle, batch, None, 82, "growing scores", patch=patch)
