"""Decode-only launches beside kernels that hold SMs for longer than the launch: the CTAs that find no SM start when others have ended,
and no unit, and no stretch of the line, may wait for theirs.  Results against the oracle."""
import numpy as np
import pytest

from paper_2609_07883_b200 import workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

HOLD_CYCLES = 300_000_000   # about 150 ms per SM held, thousands of times a launch


@pytest.mark.parametrize("form", ["fused", "two", "static"])
@pytest.mark.parametrize("heads,lens", [
    ((32, 8, 128), [300, 1500, 64, 2048, 900, 700, 1700, 250]),    # the line
    ((16, 4, 64), [9000]),
    ((8, 2, 128), [60000, 30000]),
    ((32, 4, 128), [1000] * 30 + [40000, 100]),                     # groups of eight: units, shared merges
    ((4, 4, 64), [5000, 300]),                                      # the line
    ((4, 4, 64), [20] * 432 + [5000]),                              # 433 requests: units, merged by the last ticket
    ((8, 2, 128), [20] * 432 + [60000]),                            # more than 24 units of one request: shared merges
    ((4, 2, 64), [20] * 432 + [900]),                               # every unit has a warp of its own: shared merges
])
@pytest.mark.parametrize("held", [1, 3])
def test_launches_end_although_sms_are_held(oracle, heads, lens, form, held):
    import torch

    from paper_2609_07883_b200 import binding as B

    if form == "static" and len(lens) > 256:
        pytest.skip("more requests than the static variant takes")
    shape = W.AttnShape(*heads)
    rng = np.random.default_rng(31)
    batch = W.make_batch(shape, sum(-(-x // 16) for x in lens) + 5, lens, 0, 0, rng)
    t = W.host_tensors(batch, rng)
    r = G.Runner(batch, t)
    pool = t["pool"].copy()
    assert oracle.kv_append(pool, batch, t["k_new"], t["v_new"]) == 0
    ref, ref_lse, _ = oracle.mixed_attention(pool, batch, t["q"])

    def launch():
        if form == "fused":
            r.iterate()
        elif form == "two":
            r.append()
            r.attend()
        else:
            r.append()
            B.sw_decode_attn_static(r.ctx.layout, 0, r.pool, r.dbatch, r.q, r.out, r.lse)

    launch()                                                        # loads the kernels
    torch.cuda.synchronize()
    r.out.zero_()
    r.lse.zero_()
    torch.cuda.synchronize()
    holders = [torch.cuda.Stream() for _ in range(held)]
    ends = []
    for s in holders:
        with torch.cuda.stream(s):
            torch.cuda._sleep(HOLD_CYCLES)                          # one block: one SM's shared memory is not free for a CTA
            ends.append(torch.cuda.Event())
            ends[-1].record()
    for _ in range(3):
        launch()
    done = torch.cuda.Event()
    done.record()
    done.synchronize()
    still_held = [not e.query() for e in ends]
    torch.cuda.synchronize()
    assert all(still_held), "the launch waited for the SMs that were held"
    assert r.status() == (0, 0)
    out, lse = r.results()
    G.compare(out.reshape(-1, shape.head_dim), lse.reshape(-1), ref, ref_lse, f"{form} {heads}")
