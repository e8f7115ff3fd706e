"""Performance cases of the mixed prefill-chunk + decode attention iteration.

A case is one serving iteration as a serving program runs it: decode one token for every active request and process zero
or more prefill chunks, once per layer of a stack of paged KV pools.  Every layer has its own pool and its own rows of
q / k_new / v_new / out, as in a model; the page tables, the context (workspace) and the batch are made once and shared.

Fields of a case:
    heads     query heads / KV heads / head size
    layers    layers one pass runs, one after the other on the current stream
    decodes   active requests; their contexts are the quantiles of ctx_dist between ctx_lo and ctx_hi (in a random
              order), so the total does not depend on the seed.  "uniform", or "lognormal" with median 2048, sigma 1.
    chunks    prefill chunks as "prefix+tokens" joined by commas, longest first ("" = decode-only iteration)
    call      "fused": sw_mixed_iteration_run (append and attention in one launch); "two": sw_kv_append, then
              sw_mixed_attn_run; "host": sw_mixed_iteration_host (pinned host buffers, copies inside the call)
    lse       whether the log-sum-exp of every row is asked for as well
"""
from __future__ import annotations

import math
import statistics

import numpy as np
import torch

from paper_2609_07883_b200 import binding as B
from paper_2609_07883_b200 import workloads as W

PAGE = 16
LOGNORMAL_MEDIAN, LOGNORMAL_SIGMA = 2048.0, 1.0
# the largest iteration of the repository's workloads (16 contexts of 32k-131k tokens beside 4096 tokens at prefix 98304)
MAX_KV_BYTES, MAX_FLOPS = 6.2e9, 6.7e12


def _case(name, heads, layers, decodes, ctx_dist, ctx_lo, ctx_hi, chunks, call="fused", lse=False):
    return {"name": name, "heads": heads, "layers": layers, "decodes": decodes, "ctx_dist": ctx_dist, "ctx_lo": ctx_lo,
            "ctx_hi": ctx_hi, "chunks": chunks, "call": call, "lse": lse}


def listed():
    llama = "32/8/128"
    return [
        # the smallest call: a small model with four short requests and one chunk, where launch latency is all there is
        _case("tiny", "8/2/64", 1, 4, "uniform", 64, 256, "256+128", lse=True),
        # one user alone with a medium document: a single 8k context shared by the whole device
        _case("decode_one_8k", llama, 8, 1, "uniform", 8192, 8192, ""),
        # a quiet chat server between prompts
        _case("decode_chat_16", llama, 8, 16, "uniform", 256, 2048, ""),
        # the usual chat iteration: 64 users and a chunk of somebody's prompt
        _case("chat_64_c512", llama, 8, 64, "uniform", 256, 2048, "512+512"),
        # a full batch of mixed lengths without pending prompts: bound by the KV cache
        _case("decode_mixed_128", llama, 1, 128, "lognormal", 128, 16384, ""),
        # a few long documents being answered
        _case("decode_long_4", llama, 1, 4, "uniform", 49152, 49152, ""),
        # the first chunk of a prompt on an idle server
        _case("prefill_first_2048", llama, 1, 0, "uniform", 1, 1, "0+2048"),
        # a ragged last chunk through the two-launch form, on a model with 64-element heads, log-sum-exp wanted
        _case("prefill_ragged_d64", "16/4/64", 1, 0, "uniform", 1, 1, "4111+1777", call="two", lse=True),
        # the end of two long prompts and the start of a new one in one iteration beside chat users
        _case("chunks_3_chat_64", llama, 1, 64, "uniform", 256, 2048, "28672+128,4096+128,0+256"),
        # a full batch of mixed lengths beside a chunk in the middle of a prompt
        _case("mixed_128_c1024", llama, 1, 128, "lognormal", 128, 16384, "4096+1024"),
        # long documents: the largest iteration, bound by the chunk's arithmetic
        _case("long_16_c4096", llama, 1, 16, "uniform", 32768, 131072, "98304+4096"),
        # the chat iteration of a runtime that keeps its activations on the host
        _case("host_chat_64_c512", llama, 2, 64, "uniform", 256, 2048, "512+512", call="host"),
    ]


def draw(rng):
    """One more iteration of the same ranges: the same head shapes, 0 to 256 decodes of 16 to 131072 tokens, 0 to 8 chunks of
    1 to 8192 tokens at prefixes 0 to 98304, every call form."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        heads = rng.choice(["32/8/128"] * 4 + ["16/4/64", "8/2/64", "16/8/128", "8/1/128"])
        kind = rng.choice(["decode", "prefill", "mixed", "mixed"])
        n, dist, lo, hi = 0, "uniform", 1, 1
        if kind != "prefill":
            n = log_int(1, 256)
            if rng.random() < 0.3:
                dist, lo, hi = "lognormal", 128, 16384
            else:
                lo = log_int(16, 65536)
                hi = min(131072, log_int(lo, 8 * lo))
        chunks = []
        if kind != "decode":
            k = rng.choice([1, 1, 1, 1, 2, 3, 8])
            for _ in range(k):
                chunks.append((0 if rng.random() < 0.3 else log_int(16, 98304), log_int(16, 8192 // k)))
            chunks.sort(key=lambda c: -(2 * c[0] + c[1]) * c[1])
        case = _case("", heads, 1, n, dist, lo, hi, ",".join("%d+%d" % c for c in chunks),
                     call=rng.choice(["fused", "fused", "fused", "two", "host"]), lse=rng.random() < 0.25)
        del case["name"]
        one = work(case)
        if one["bytes"] > MAX_KV_BYTES or one["flops"] > MAX_FLOPS:
            continue
        if one["bytes"] < 3e8 and one["flops"] < 5e10:
            case["layers"] = rng.randint(1, 8)
        return case


def _shape(case):
    hq, hkv, d = (int(x) for x in case["heads"].split("/"))
    return W.AttnShape(hq, hkv, d)


def _chunks(case):
    return [tuple(int(x) for x in c.split("+")) for c in case["chunks"].split(",") if c]


def _contexts(case):
    n, lo, hi = case["decodes"], case["ctx_lo"], case["ctx_hi"]
    at = (np.arange(n) + 0.5) / max(n, 1)
    if case["ctx_dist"] == "lognormal":
        z = np.array([statistics.NormalDist().inv_cdf(float(u)) for u in at])
        lens = np.clip(np.floor(LOGNORMAL_MEDIAN * np.exp(LOGNORMAL_SIGMA * z)), lo, hi)
    else:
        lens = np.floor(lo + at * (hi - lo + 1))
    return lens.astype(np.int32)


def work(case):
    """Each layer reads the K/V rows its requests attend once, q and the new K/V rows once, and writes out, the new rows
    and (if asked for) the log-sum-exp once; the page tables are read once per layer.  Two multiply-adds per (query head,
    attended key, element)."""
    sh, chunks, lens = _shape(case), _chunks(case), _contexts(case).astype(np.int64)
    rows = sum(c for _, c in chunks) + len(lens)
    cached = int(lens.sum()) - len(lens) + sum(p for p, _ in chunks)       # rows that are in the pool before the pass
    new = 2 * rows * sh.token_bytes                                        # the iteration's rows: read, and written to the pool
    io = 2 * rows * sh.num_q_heads * sh.head_dim * 2 + (4 * rows * sh.num_q_heads if case["lse"] else 0)
    tables = 4 * (sum(-(-int(x) // PAGE) for x in lens) + sum(-(-(p + c) // PAGE) for p, c in chunks) + 2 * len(lens) + 1)
    keys = int(lens.sum()) + sum(c * p + c * (c + 1) // 2 for p, c in chunks)
    return {"bytes": case["layers"] * (cached * sh.token_bytes + new + io + tables),
            "flops": case["layers"] * 4 * sh.num_q_heads * sh.head_dim * keys}


def _inputs(case, seed):
    """The iteration's batch (page tables, lengths) and, per layer, the pool with its cached rows, the new rows and the
    queries: N(0,1) in bf16, as normalised activations are, with randomly scattered pages."""
    rng = np.random.Generator(np.random.PCG64(seed))
    sh, chunks, lens = _shape(case), _chunks(case), rng.permutation(_contexts(case))
    need = sum(-(-int(x) // PAGE) for x in lens) + sum(-(-(p + c) // PAGE) for p, c in chunks)
    num_pages = need + 64                                                  # some free pages, as any pool has
    if len(chunks) <= 1:
        P, C = chunks[0] if chunks else (0, 0)
        batch = W.make_batch(sh, num_pages, lens, P, C, rng)
    else:
        batch = W.make_multi_batch(sh, num_pages, lens, chunks, rng)
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    rows, layers = batch.num_rows, case["layers"]

    def normal(*size):
        return torch.empty(*size, dtype=torch.bfloat16, device=dev).normal_(generator=gen)

    return need, batch, {
        "pools": [normal(num_pages * sh.page_elems) for _ in range(layers)],
        "q": [normal(rows, sh.num_q_heads, sh.head_dim) for _ in range(layers)],
        "k_new": [normal(rows, sh.num_kv_heads, sh.head_dim) for _ in range(layers)],
        "v_new": [normal(rows, sh.num_kv_heads, sh.head_dim) for _ in range(layers)],
    }


def prepare(case, seed):
    """A serving program's state before the call: the inputs, the output buffers, the batch on the device, the context."""
    need, batch, state = _inputs(case, seed)
    sh, dev = _shape(case), state["q"][0].device
    rows, layers = batch.num_rows, case["layers"]
    state["call"] = case["call"]
    state["ctx"] = B.Context(sh, need + 64, max(batch.chunk_len, 1), max(batch.num_decode, 1), need + 16, device=dev.index)
    state["out"] = [torch.zeros(rows, sh.num_q_heads, sh.head_dim, dtype=torch.bfloat16, device=dev) for _ in range(layers)]
    state["lse"] = [torch.zeros(rows, sh.num_q_heads, dtype=torch.float32, device=dev) if case["lse"] else None
                    for _ in range(layers)]
    if case["call"] == "host":
        for name in ("q", "k_new", "v_new", "out", "lse"):
            state[name] = [None if t is None else t.cpu().pin_memory() for t in state[name]]
        state["batch"], state["keep"] = B.host_batch_struct(batch)
    else:
        state["batch"] = B.DeviceBatch(batch, dev)
    return state


def run(state):
    """One iteration over the layer stack."""
    ctx, batch, call = state["ctx"], state["batch"], state["call"]
    for pool, q, k, v, out, lse in zip(state["pools"], state["q"], state["k_new"], state["v_new"], state["out"], state["lse"]):
        if call == "fused":
            B.sw_mixed_iteration_run(ctx, pool, batch, k, v, q, out, lse)
        elif call == "two":
            B.sw_kv_append(ctx, pool, batch, k, v)
            B.sw_mixed_attn_run(ctx, pool, batch, q, out, lse)
        else:
            B.sw_mixed_iteration_host(ctx, pool, batch, q, k, v, out, lse)
    return {"out": state["out"], "pools": state["pools"], "lse": [t for t in state["lse"] if t is not None]}


def tolerance(case):
    """Softmax weights and outputs are rounded to bf16 (2^-9 each); sums and maxima are fp32.  Against the same attention in
    fp64, on rows sampled from every listed case and six drawn ones, the outputs are off by 2.4e-3 at most in the 2-norm
    and by 0.013 in the largest element: about four times that is stated.  (The pools hold copies: exact.)"""
    return {"rel": 1e-2, "max": 0.06}


def _attend(q, k, v, scale, causal_from):
    """64-bit attention of q [rows, heads, d] over k / v [keys, kv heads, d]; row i sees keys [0, causal_from + i].
    Returns (out [rows, heads, d], lse [rows, heads])."""
    rows, hq, d = q.shape
    keys, hkv, _ = k.shape
    g = hq // hkv
    out, lse = torch.empty(rows, hq, d, dtype=torch.float64, device=q.device), torch.empty(rows, hq, dtype=torch.float64, device=q.device)
    step = max(1, int(2.5e8) // (keys * g))                                # rows at a time: about 2 GB of scores
    at = torch.arange(keys, device=q.device)
    for h in range(hkv):
        kh, vh = k[:, h].double().t().contiguous(), v[:, h].double().contiguous()
        for r0 in range(0, rows, step):
            n = min(step, rows - r0)
            s = (q[r0:r0 + n, h * g:(h + 1) * g].double().reshape(n * g, d) @ kh).mul_(scale).view(n, g, keys)
            first = causal_from + r0 + 1                                   # earlier keys are seen by every one of these rows
            seen = at[first:] <= causal_from + r0 + torch.arange(n, device=q.device)[:, None]
            s[:, :, first:].masked_fill_(~seen[:, None, :], -math.inf)
            m = s.amax(-1, keepdim=True)
            s.sub_(m).exp_()
            total = s.sum(-1, keepdim=True)
            out[r0:r0 + n, h * g:(h + 1) * g] = (s.view(n * g, keys) @ vh).view(n, g, d) / total
            lse[r0:r0 + n, h * g:(h + 1) * g] = (m + total.log()).squeeze(-1)
    return out, lse


def exact(case, seed):
    """The same iteration as plain torch gives it in 64 bits: every request's rows are put into its pages, its keys and
    values gathered, and ordinary softmax attention done.  (The pools hold copies and stay bf16.)"""
    _, batch, given = _inputs(case, seed)
    sh, chunks = _shape(case), _chunks(case)
    spans, row, page = [], 0, 0                                            # (first row, rows, first position, pages)
    for p, c in chunks:
        n = -(-(p + c) // PAGE)
        spans.append((row, c, p, batch.prefill_pages[page:page + n]))
        row, page = row + c, page + n
    for i, x in enumerate(batch.decode_kv_len):
        pages = batch.decode_pages[batch.decode_page_indptr[i]:batch.decode_page_indptr[i + 1]]
        spans.append((row + i, 1, int(x) - 1, pages))
    result = {"out": [], "pools": given["pools"], "lse": []}
    for pool, q, k_new, v_new in zip(given["pools"], given["q"], given["k_new"], given["v_new"]):
        pages_of = pool.view(-1, 2, sh.num_kv_heads, PAGE, sh.head_dim)
        out = torch.empty(q.shape, dtype=torch.float64, device=q.device)
        lse = torch.empty(q.shape[:2], dtype=torch.float64, device=q.device)
        for r, n, first, pages in spans:
            ids = torch.from_numpy(np.ascontiguousarray(pages).astype(np.int64)).to(q.device)
            pos = torch.arange(first, first + n, device=q.device)
            pages_of[ids[pos // PAGE], 0, :, pos % PAGE] = k_new[r:r + n]
            pages_of[ids[pos // PAGE], 1, :, pos % PAGE] = v_new[r:r + n]
            kv = pages_of[ids].permute(1, 0, 3, 2, 4).reshape(2, -1, sh.num_kv_heads, sh.head_dim)[:, :first + n]
            out[r:r + n], lse[r:r + n] = _attend(q[r:r + n], kv[0], kv[1], sh.head_dim ** -0.5, first)
        result["out"].append(out)
        if case["lse"]:
            result["lse"].append(lse)
    return result
