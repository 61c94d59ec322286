"""Performance cases of the agx library: what an agent runtime built on it has it do, through ``agx.py``.

A pass of a *step* case is one forward step of a model: ``attn_prefixed_append`` for every layer (each layer with K/V
pools of its own, as a model has them), then ``accept_greedy`` over the logits of the verify rows (one row for a block that
is prefilled).  A *host* case is the same step for activations that live in pinned host memory.  A *setup* case is what
happens once when a request arrives: its n-gram draft table, the first drafts, and private copies of cut pages.

Blocks are written ``count x prefix + q``: ``"4x32768+8,1x30720+2048"`` is four verify blocks of 8 rows behind 32768
cached tokens and one 2048-row suffix behind 30720.  Values are N(0, 1), page tables are shuffled, drafts are accepted
token by token with probability 1/4 (the rate the paper reports).
"""
import math

import numpy as np
import torch

from paper_2605_10380_b200 import agx
from paper_2605_10380_b200 import workloads as W

PAGE = 16
VERIFY_ROWS = 16   # blocks of up to this many rows are decode or verify blocks (logits for every row); longer ones are prefill


def _step(name, blocks, layers, hq=32, hkv=8, d=128, dtype="bf16", vocab=128256, logits="bf16", shared=0, kind="step"):
    c = dict(kind=kind, blocks=blocks, layers=layers, hq=hq, hkv=hkv, d=d, dtype=dtype, vocab=vocab, logits=logits, shared=shared)
    return dict(name=name, **c) if name else c


def _setup(name, tokens, n, seqs, k, pages, layers, hq=32, hkv=8, d=128):
    c = dict(kind="setup", tokens=tokens, n=n, seqs=seqs, k=k, pages=pages, layers=layers, hq=hq, hkv=hkv, d=d, dtype="bf16")
    return dict(name=name, **c) if name else c


def listed():
    p4, q4 = W.c4_lengths()
    ragged = ",".join(f"1x{int(p)}+{int(q)}" for p, q in zip(p4, q4))
    return [
        # the smallest verify step, fp32 (the tiny configuration): launches and latency only
        _step("tiny_verify_f32", "1x256+4", 1, hq=4, hkv=2, d=64, dtype="f32", vocab=1024, logits="f32"),
        # one agent, token by token: the fall-back when the draft table has nothing, a 32-layer model
        _step("decode_4k", "1x4096+1", 32),
        # one agent verifying 7 drafts, a 32-layer model (the decode-verification configuration)
        _step("verify_4k", "1x4096+8", 32),
        # a server decoding for 16 agents with ragged contexts
        _step("decode_batch", "3x2051+1,3x3600+1,4x4580+1,2x6007+1,2x9123+1,2x14264+1", 4),
        # a server verifying for 16 agents (the benchmark's serving batch)
        _step("verify_batch", "16x8192+8", 2),
        # planner prompt with a cached prefix (the prefix-cached-prefill configuration)
        _step("prefill_cached", "1x3072+512", 8, hq=24),
        # the agent's second, shorter model call
        _step("prefill_short", "1x1000+128", 8),
        # the same planner prompt with nothing cached
        _step("prefill_cold", "1x0+3584", 2, hq=24),
        # mixed batch: 8 verify blocks and 8 suffix prefills behind a shared 2048-token prefix
        _step("ragged_mixed", ragged, 1, shared=2048),
        # the long-context configuration, the largest step
        _step("long_context", "4x32768+8,1x30720+2048", 1),
        # verify_4k for a runtime whose activations are host buffers
        _step("host_verify_4k", "1x4096+8", 32, kind="host"),
        # a request arrives: trigram table over its prompt, first drafts, cut pages copied in 8 layer pools
        _setup("request_setup", 4096, 3, 16, 4, 16, 8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fits(c):
    w = work(c)
    return w["flops"] <= 1.0e12 and w["bytes"] <= 8.0e8


def draw(rng):
    kind = rng.choice(["tiny", "decode", "verify", "decode_batch", "verify_batch", "cached", "short", "cold", "mixed", "long", "host",
                       "setup"])
    while True:
        hq, hkv = rng.choice([(32, 8), (32, 8), (32, 8), (24, 8), (24, 8), (40, 8), (16, 2)])
        if kind == "tiny":
            c = _step("", f"1x{_log(rng, 20, 1500)}+{rng.randint(1, 8)}", 1, hq=rng.choice([4, 8]), hkv=2, d=rng.choice([64, 128]),
                      dtype="f32", vocab=_log(rng, 500, 33000), logits="f32")
        elif kind == "decode":
            c = _step("", f"1x{_log(rng, 200, 60000)}+1", rng.randint(4, 32), hq, hkv, vocab=rng.choice([32000, 32003, 128256]))
        elif kind == "verify":
            c = _step("", f"1x{_log(rng, 200, 60000)}+{rng.randint(2, 16)}", rng.randint(4, 32), hq, hkv, vocab=rng.choice([32000, 128256]),
                      logits=rng.choice(["bf16", "f32"]))
        elif kind == "decode_batch":
            c = _step("", ",".join(f"1x{_log(rng, 300, 16384)}+1" for _ in range(_log(rng, 2, 48))), rng.randint(1, 4), hq, hkv)
        elif kind == "verify_batch":
            c = _step("", ",".join(f"1x{_log(rng, 300, 16384)}+{rng.randint(1, 16)}" for _ in range(_log(rng, 2, 32))), rng.randint(1, 4), hq, hkv,
                      logits=rng.choice(["bf16", "f32"]))
        elif kind == "cached":
            c = _step("", f"1x{_log(rng, 1024, 16000)}+{_log(rng, 256, 1500)}", rng.randint(2, 8), hq, hkv)
        elif kind == "short":
            c = _step("", f"1x{_log(rng, 300, 3000)}+{_log(rng, 40, 256)}", rng.randint(4, 12), hq, hkv)
        elif kind == "cold":
            c = _step("", f"{rng.randint(1, 2)}x0+{_log(rng, 256, 5000)}", rng.randint(1, 4), hq, hkv)
        elif kind == "mixed":
            v = [f"1x{_log(rng, 2048, 16384)}+{rng.choice([1, 2, 4, 8, 16])}" for _ in range(rng.randint(2, 8))]
            f = [f"1x{_log(rng, 2048, 16384)}+{rng.randint(128, 1024)}" for _ in range(rng.randint(1, 8))]
            c = _step("", ",".join(v + f), 1, hq, hkv, shared=2048)
        elif kind == "long":
            c = _step("", f"{rng.randint(1, 4)}x{_log(rng, 16384, 40000)}+{rng.randint(1, 12)},1x{_log(rng, 8192, 40000)}+{_log(rng, 512, 2048)}", 1, hq, hkv)
        elif kind == "host":
            c = _step("", f"1x{_log(rng, 300, 16384)}+{rng.choice([1, 4, 8, 11, 96, 500])}", rng.randint(4, 16), hq, hkv, kind="host")
        else:
            c = _setup("", _log(rng, 300, 40000), rng.choice([2, 3]), rng.randint(1, 64), rng.randint(1, 8), rng.randint(1, 32),
                       rng.randint(1, 16), hq, hkv)
        if _fits(c):
            return c


def _blocks(case):
    P, Q = [], []
    for part in case["blocks"].split(","):
        n, rest = part.split("x")
        p, q = rest.split("+")
        P += [int(p)] * int(n)
        Q += [int(q)] * int(n)
    return np.asarray(P, np.int32), np.asarray(Q, np.int32)


def work(case):
    es = 2 if case["dtype"] == "bf16" else 4
    row = case["hkv"] * case["d"] * es   # one token's K (or V)
    if case["kind"] == "setup":
        # the prompt once, the drafts, every copied page read and written; (the table itself is internal)
        return {"bytes": 4 * case["tokens"] + 4 * case["seqs"] * (case["k"] * 2 + case["n"]) + case["layers"] * case["pages"] * 4 * PAGE * row,
                "flops": 0}
    P, Q = (a.astype(np.int64) for a in _blocks(case))
    kv_tokens = int((P + Q).sum()) - case["shared"] * (len(P) - 1 if case["shared"] else 0)
    # cached K/V once, the block's K/V read and written, Q in, the result out
    per_layer = 2 * row * kv_tokens + 2 * row * int(Q.sum()) + 2 * int(Q.sum()) * case["hq"] * case["d"] * es
    rows = int(sum(q if q <= VERIFY_ROWS else 1 for q in Q))
    return {"bytes": case["layers"] * per_layer + rows * case["vocab"] * (2 if case["logits"] == "bf16" else 4),
            "flops": case["layers"] * 4 * case["d"] * case["hq"] * int((Q * P + Q * (Q + 1) // 2).sum())}


def tolerance(case):
    if case["kind"] == "setup":
        return "exact"
    if case["dtype"] == "f32":
        return {"rel": 2e-6, "max": 1e-5}   # measured against fp64: rel 2.6e-7, max 1.1e-6; other orders of the sums
    return {"rel": 1e-2, "max": 1.5e-1}     # measured against fp64: rel 2.0e-3 to 2.4e-3, max 0.006 to 0.038 (nothing cached)


def _normal(gen, dtype, *shape):
    return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.bfloat16 if dtype == "bf16" else torch.float32)


def _prepare_setup(case, seed, s, gen, rng):
    # a prompt made of phrases that come back (instructions, examples, tool descriptions), with fresh tokens in between
    phrases = [rng.integers(0, 32000, size=int(rng.integers(4, 40))) for _ in range(24)]
    parts, n = [], 0
    while n < case["tokens"]:
        parts.append(phrases[int(rng.integers(0, len(phrases)))] if rng.random() < 0.7 else rng.integers(0, 32000, size=8))
        n += len(parts[-1])
    stream = np.concatenate(parts)[:case["tokens"]].astype(np.int32)
    m = case["n"] - 1
    at = rng.integers(0, case["tokens"] - m, size=case["seqs"])
    s["stream"] = torch.from_numpy(stream).cuda()
    s["context"] = torch.from_numpy(np.stack([stream[a:a + m] for a in at])).cuda()
    s["fill"] = torch.from_numpy(rng.integers(0, 32000, size=(case["seqs"], case["k"])).astype(np.int32)).cuda()
    s["drafts"] = torch.zeros(case["seqs"], case["k"], dtype=torch.int32, device="cuda")
    s["has"] = torch.zeros(case["seqs"], dtype=torch.int32, device="cuda")
    s["lut"] = torch.empty(agx.ngram_lut_bytes(case["tokens"]), dtype=torch.uint8, device="cuda")
    s["lut_ws"] = torch.empty(agx.ngram_workspace_bytes(case["tokens"]), dtype=torch.uint8, device="cuda")
    pages = 3 * case["pages"] + 5
    perm = rng.permutation(pages).astype(np.int32)
    s["src"] = torch.from_numpy(perm[:case["pages"]]).cuda()
    s["dst"] = torch.from_numpy(perm[case["pages"]:2 * case["pages"]]).cuda()
    s["k_pools"] = _normal(gen, "bf16", case["layers"], pages, case["hkv"], PAGE, case["d"])
    s["v_pools"] = _normal(gen, "bf16", case["layers"], pages, case["hkv"], PAGE, case["d"])
    s["k_layers"], s["v_layers"] = list(s["k_pools"]), list(s["v_pools"])
    return s


def _logits(case, gen, rng, rows, drafted):
    """Logits whose winners are planted, and drafts that meet them with probability 1/4 each (``drafted``: rows with a draft behind them)."""
    dt = torch.bfloat16 if case["logits"] == "bf16" else torch.float32
    logits = torch.randn(rows, case["vocab"], generator=gen, device="cuda", dtype=dt)
    target = rng.integers(0, case["vocab"], size=rows)
    logits[torch.arange(rows, device="cuda"), torch.from_numpy(target).cuda()] = 8.0
    drafts = [int(target[r]) if rng.random() < 0.25 else int(rng.integers(0, case["vocab"])) for r in drafted]
    return logits, torch.tensor(drafts or [0], dtype=torch.int32)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rng = np.random.default_rng(seed)
    h = agx.Handle(case["hq"], case["hkv"], case["d"], case["dtype"])
    s = {"case": case, "h": h}
    if case["kind"] == "setup":
        return _prepare_setup(case, seed, s, gen, rng)
    hq, hkv, d, layers, dtype = case["hq"], case["hkv"], case["d"], case["layers"], case["dtype"]
    s["P"], s["Q"] = P, Q = _blocks(case)
    total_q = int(Q.sum())
    table, pages = W.build_page_table(rng, P.astype(np.int64) + Q, case["shared"], spare_pages=7)
    s["table"] = torch.from_numpy(table).cuda()
    s["k_pools"] = torch.empty(layers, pages, hkv, PAGE, d, device="cuda", dtype=torch.bfloat16 if dtype == "bf16" else torch.float32)
    s["v_pools"] = torch.empty_like(s["k_pools"])
    for pool in (s["k_pools"], s["v_pools"]):
        for l in range(layers):
            pool[l] = _normal(gen, dtype, pages, hkv, PAGE, d)
    s["k_layers"], s["v_layers"] = list(s["k_pools"]), list(s["v_pools"])   # a program has its layers' tensors at hand
    q = _normal(gen, dtype, layers, total_q, hq, d)
    k_new = _normal(gen, dtype, layers, total_q, hkv, d)
    v_new = _normal(gen, dtype, layers, total_q, hkv, d)
    # the accept step: every row of a decode or verify block, the last row of a prefilled one
    rows = np.asarray([n if n <= VERIFY_ROWS else 1 for n in Q], np.int32)
    cu = W.cu_from_q(rows)
    drafted = [int(r) for b in range(len(rows)) for r in range(cu[b], cu[b + 1] - 1)]
    logits, drafts = _logits(case, gen, rng, int(cu[-1]), drafted)
    if case["kind"] == "host":
        pin = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)  # noqa: E731
        s["q"], s["k_new"], s["v_new"], s["logits"], s["drafts"] = (pin(t) for t in (q, k_new, v_new, logits, drafts))
        s["q"], s["k_new"], s["v_new"] = list(s["q"]), list(s["k_new"]), list(s["v_new"])
        s["out"] = torch.zeros(layers, total_q, hq, d, dtype=q.dtype).pin_memory()
        s["out_layers"] = list(s["out"])
        s["acc"], s["nxt"], s["seq_lens"] = (torch.zeros(len(P), dtype=torch.int32).pin_memory() for _ in range(3))
        with_accept = bool((rows == Q).all())   # (the host step's acceptance covers every row of its blocks)
        s["vocab"] = [0] * (layers - 1) + [case["vocab"] if with_accept else 0]
        n = max(h.verify_step_host_workspace_bytes(P, Q, case["logits"], case["vocab"], v) for v in set(s["vocab"]))
        s["ws"] = torch.empty(n, dtype=torch.uint8, device="cuda")
        return s
    s.update(q=list(q), k_new=list(k_new), v_new=list(v_new), logits=logits, drafts=drafts.cuda(), out=torch.zeros_like(q), cu=torch.from_numpy(cu).cuda(),
             acc=torch.zeros(len(P), dtype=torch.int32, device="cuda"), nxt=torch.zeros(len(P), dtype=torch.int32, device="cuda"),
             argmax=torch.zeros(int(cu[-1]), dtype=torch.int32, device="cuda"),
             # committed lengths: a prefill's last row stands for the whole block
             seq_lens=torch.from_numpy((P + Q - rows).astype(np.int32)).cuda())
    s["out_layers"] = list(s["out"])
    # every layer has pools of its own and the cached prefix was written by earlier steps
    h.set_option(agx.AGX_OPT_EARLY_PREFIX_LOADS, 1)
    n = h.attn_workspace_bytes(P, Q)
    s["ws"] = torch.empty(n, dtype=torch.uint8, device="cuda") if n else None
    s["accept_ws"] = torch.empty(h.accept_workspace_bytes(int(cu[-1]), case["vocab"]), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    case, h = s["case"], s["h"]
    k_pools, v_pools = s["k_layers"], s["v_layers"]
    if case["kind"] == "setup":
        h.ngram_build(s["stream"], case["n"], s["lut"], s["lut_ws"])
        h.ngram_draft(s["lut"], s["context"], s["fill"], case["k"], s["drafts"], s["has"])
        for l in range(case["layers"]):
            h.kv_copy_pages(k_pools[l], v_pools[l], s["src"], s["dst"])
        return {"drafts": s["drafts"], "has_draft": s["has"], "k_pools": s["k_pools"], "v_pools": s["v_pools"]}
    q, k_new, v_new, out = s["q"], s["k_new"], s["v_new"], s["out_layers"]
    if case["kind"] == "host":
        for l, vocab in enumerate(s["vocab"]):
            h.verify_step_host(k_pools[l], v_pools[l], s["table"], s["P"], s["Q"], q[l], k_new[l], v_new[l], s["logits"], case["logits"],
                               case["vocab"], vocab, s["drafts"], out[l], s["acc"], s["nxt"], s["seq_lens"], s["ws"], enqueue_only=True)
        torch.cuda.current_stream().synchronize()   # the results are host buffers: a program waits before it reads them
        return {"out": s["out"], "accept_len": s["acc"], "next_token": s["nxt"], "seq_lens": s["seq_lens"], "k_pools": s["k_pools"],
                "v_pools": s["v_pools"]}
    for l in range(case["layers"]):
        h.attn_prefixed_append(q[l], k_new[l], v_new[l], k_pools[l], v_pools[l], s["table"], s["P"], s["Q"], out[l], None, s["ws"])
    h.accept_greedy(s["logits"], case["logits"], case["vocab"], s["drafts"], s["cu"], s["acc"], s["nxt"], s["argmax"], s["seq_lens"],
                    s["accept_ws"])
    return {"out": s["out"], "accept_len": s["acc"], "next_token": s["nxt"], "argmax": s["argmax"], "seq_lens": s["seq_lens"],
            "k_pools": s["k_pools"], "v_pools": s["v_pools"]}
