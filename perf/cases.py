"""Performance cases: what a serving program asks of this library, one dict of plain values per case.

A case's "kind" is one of
  step         a whole greedy verify step: ancestor masks, attention of every layer (one call per layer, as a
               decoder issues them, or all layers in one call), then LM head + acceptance + compaction
  attention    the attention calls alone (a decoder with a tail of its own)
  lmhead       the LM-head arg-max alone
  topk         the tail at a sampling temperature for top-k trees (one fused call)
  chain_q      the tail at a temperature for chains sampled from the draft's distributions (three calls)
  tree_q       the tail at a temperature for trees whose children were sampled (three calls)
  draft        the draft side's feature aggregation

Inputs are drawn on the GPU from the seed alone: standard-normal K and V, scores with a standard deviation of
about 2, and hidden states that give every LM-head row a dozen likely tokens well above the bulk of the vocabulary,
so that drafts are accepted over several levels and then rejected, as with trained models.
"""
import math
import random

import numpy as np
import torch

from paper_2509_18824_b200 import binding as sd
from paper_2509_18824_b200 import workloads as wl

N_CAND = 12                       # likely tokens planted behind every tree node
INV_TEMP = 1.0 / 0.8

# a 7B-class GQA decoder, as in the repository's configurations
MODEL = dict(Hq=28, Hkv=4, Hd=3584, V=152064, L=28)


def _case(name, kind, **kw):
    c = dict(name=name, kind=kind, B=1, T=60, tree="eagle", depth=6, prefix_lo=2048, prefix_hi=2048, shuffled=False,
             ragged_nodes=False, one_call=False, graph=False, **MODEL)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest whole step: one short sequence, a tree of eight nodes, one small layer; launches and host calls
        _case("tiny_step", "step", T=8, tree="tiny", depth=3, prefix_lo=128, prefix_hi=128, Hq=4, Hkv=1, Hd=256, V=1024, L=1),
        # one user's decoding step: 28 dependent layers of little work each, issued call by call
        _case("single_user_step", "step", shuffled=True),
        # the headline step of the benchmark: 8 sequences, prefix 4096, replayed from a CUDA graph
        _case("batch_step", "step", B=8, prefix_lo=4096, prefix_hi=4096, graph=True),
        # a busy server: 16 sequences of very different lengths in a shuffled pool, trees of different sizes
        _case("ragged_step", "step", B=16, prefix_lo=512, prefix_hi=16384, shuffled=True, ragged_nodes=True),
        # chain decoding, the paper's own setting (root + 10 drafts): bound by the K/V stream
        _case("chain_step", "step", B=8, T=11, tree="chain", depth=10, prefix_lo=4096, prefix_hi=4096, graph=True),
        # short trees, every layer's attention in one call (inputs of all layers on hand)
        _case("short_tree_layers", "attention", B=8, T=28, depth=5, prefix_lo=4096, prefix_hi=4096, one_call=True),
        # long multimodal contexts, a few layers, one call per layer
        _case("long_context_attention", "attention", B=4, prefix_lo=8192, prefix_hi=8192, L=4),
        # the tail of the benchmark's step at a sampling temperature, top-k trees
        _case("topk_sampled_tail", "topk", B=8, prefix_lo=1000, prefix_hi=4096),
        # the tail of chain decoding at a temperature: W is streamed for 88 rows
        _case("chain_sampled_tail", "chain_q", B=8, T=11, tree="chain", depth=10, prefix_lo=1000, prefix_hi=4096),
        # the tail for trees whose children were sampled, on the benchmark's batch
        _case("tree_sampled_tail", "tree_q", B=8, prefix_lo=1000, prefix_hi=4096),
        # draft side, prefill: the features of 4096 tokens
        dict(name="draft_prefill", kind="draft", S=4096, L=28, Q=4, H=28, same=False),
        # draft side, decoding: the features of the tokens a step accepted, un-projected (K and V one buffer)
        dict(name="draft_decode", kind="draft", S=37, L=28, Q=4, H=28, same=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "attention", "attention", "lmhead", "topk", "chain_q", "tree_q", "draft"])
    if kind == "draft":
        return dict(kind="draft", S=_log(rng, 1, 4096), L=rng.randint(8, 32), Q=rng.randint(1, 8), H=rng.choice([8, 16, 28]),
                    same=rng.random() < 0.5)
    heads = rng.choice([(28, 4), (28, 4), (32, 8), (16, 2), (8, 1), (16, 4)])
    V, Hd = rng.choice([(152064, 3584), (152064, 3584), (128256, 4096), (32000, 4096), (50257, 2048), (4099, 1024)])
    chain = kind == "chain_q" or (kind != "tree_q" and kind != "topk" and rng.random() < 0.3)
    B = _log(rng, 1, 16)
    T = rng.randint(2, 17) if chain else rng.randint(9, 64)
    hi = _log(rng, 60, 16384)
    while B * hi > 65536:
        hi //= 2
    lo = hi if rng.random() < 0.5 else max(16, hi // rng.randint(2, 16))
    if kind in ("topk", "chain_q", "tree_q"):
        B, hi, lo = min(B, 512 // T), min(hi, 4096), min(lo, 4096)
    return dict(kind=kind, B=B, T=T, tree="chain" if chain else "eagle", depth=T - 1 if chain else rng.randint(3, min(7, T - 2)),
                prefix_lo=lo, prefix_hi=hi, shuffled=rng.random() < 0.7, ragged_nodes=rng.random() < 0.4,
                one_call=rng.random() < 0.25, graph=rng.random() < 0.5, Hq=heads[0], Hkv=heads[1], Hd=Hd, V=V,
                L=rng.choice([1, 2, 4, 12, 28]))


# ---------------------------------------------------------------------------------------------- inputs
def _gen(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1000003 + sum((i + 1) * ord(ch) for i, ch in enumerate(what))) & 0x7FFFFFFF)
    return g


def _randn(seed, what, shape, scale=1.0, dtype=torch.bfloat16):
    x = torch.empty(shape, dtype=dtype, device="cuda").normal_(generator=_gen(seed, what))
    return x.mul_(scale) if scale != 1.0 else x


def _trees(c, seed):
    """Lengths, node counts, parent arrays and block table of the batch (numpy)."""
    rng = random.Random(seed * 7919 + 17)
    g = np.random.default_rng([seed, 5])
    B, T = c["B"], c["T"]
    # lengths spread evenly over the range, in an order of the seed's (the pool then has one size for every seed)
    lens = np.array([c["prefix_lo"] + int((c["prefix_hi"] - c["prefix_lo"]) * (i + 0.5) / B) for i in range(B)], np.int32)
    g.shuffle(lens)
    n_nodes = np.full(B, T, np.int32)
    parents = np.zeros((B, T), np.int32)
    for b in range(B):
        if c["tree"] == "tiny":
            parents[b] = wl.TINY_PARENTS
            continue
        # trees of one batch differ: depth by one around the case's, node count down to half where ragged
        n = rng.randint(max(2, T // 2), T) if c["ragged_nodes"] else T
        if c["tree"] == "chain":
            parents[b, :n] = wl.chain_tree(n)
        else:
            depth = max(2, min(c["depth"] + rng.choice([-1, 0, 0, 1]), n - 1))
            parents[b, :n] = wl.eagle_style_tree(g, n, depth)
        n_nodes[b] = n
    need = (lens.astype(np.int64) + T + wl.BLOCK - 1) // wl.BLOCK
    n_blocks = int(need.sum()) + 3
    pool = g.permutation(n_blocks) if c["shuffled"] else np.arange(n_blocks)
    table = np.zeros((B, int(need.max())), np.int32)
    at = 0
    for b in range(B):
        table[b, :need[b]] = pool[at:at + need[b]]
        at += int(need[b])
    return lens, n_nodes, parents, table, n_blocks


def _lm_inputs(s, c, seed, parents, n_nodes):
    """LM-head weights, hidden states with likely tokens, and draft tokens taken from those (top-k children in
    order of likelihood; now and then the draft model misses the most likely one)."""
    M, Hd, V = s["M"], c["Hd"], c["V"]
    B, T = c["B"], c["T"]
    W = _randn(seed, "W", (V, Hd), 1.0 / math.sqrt(Hd))
    g = _gen(seed, "tokens")
    first = torch.randint(0, V, (M, 1), device="cuda", generator=g)
    cand = (first + torch.arange(N_CAND, device="cuda")[None] * (V // (N_CAND + 1))) % V          # distinct
    level = math.log(V) + 4.0 - 0.7 * torch.arange(N_CAND, device="cuda", dtype=torch.float32)
    hidden = _randn(seed, "hidden", (M, Hd), dtype=torch.float32)
    for k in range(N_CAND):
        hidden.add_(W[cand[:, k]].float() * level[k])
    miss = (torch.rand((M,), device="cuda", generator=g) < 0.2).long()
    par = torch.from_numpy(parents).long()
    rank = torch.zeros((B, T), dtype=torch.long)                                                # place among the siblings
    for b in range(B):
        seen = {}
        for j in range(1, int(n_nodes[b])):
            p = int(parents[b, j])
            rank[b, j] = seen.get(p, 0)
            seen[p] = int(rank[b, j]) + 1
    row = (torch.arange(B)[:, None] * T + par.clamp(min=0)).cuda()
    pick = (rank.cuda() + miss[row]).clamp(max=N_CAND - 1)
    s["W"], s["hidden"] = W, hidden.to(torch.bfloat16)
    s["draft"] = cand[row.reshape(-1)].gather(1, pick.reshape(-1, 1)).reshape(B, T).to(torch.int32).contiguous()
    s["cand"], s["level"], s["rank"], s["row"] = cand, level, rank, row


def _q_inputs(s, c, seed):
    """Draft distributions near the target's, children drawn from their parent's."""
    M, V, B, T = s["M"], c["V"], c["B"], c["T"]
    g = _gen(seed, "q")
    q = torch.empty((M, V), device="cuda").normal_(generator=g)
    q.scatter_add_(1, s["cand"], s["level"] + 0.8 * torch.empty((M, N_CAND), device="cuda").normal_(generator=g))
    q = torch.softmax(q.mul_(INV_TEMP), dim=1)
    rank, row = s["rank"].cuda(), s["row"]
    tok = s["draft"]
    for k in range(int(rank.max()) + 1):                      # the k-th child of every node: one draw per LM-head row
        u = torch.rand((M, V), device="cuda", generator=g).clamp_(min=1e-12)
        drawn = (q.log() - torch.log(-torch.log(u))).argmax(dim=1).to(torch.int32)
        tok = torch.where(rank == k, drawn[row], tok)
    s["draft"] = tok.contiguous()
    s["q_rows"] = q.view(B, T, V)
    s["q_tok"] = q[row.reshape(-1)].gather(1, tok.long().reshape(-1, 1)).reshape(B, T).contiguous()


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "draft":
        D = c["H"] * 128
        k = _randn(seed, "k", (c["S"], c["L"], D))
        return dict(c=c, qp=_randn(seed, "qp", (c["Q"], D), 2.0), k=k, v=k if c["same"] else _randn(seed, "v", (c["S"], c["L"], D)),
                    out=torch.empty((c["S"], c["Q"], D), dtype=torch.bfloat16, device="cuda"))
    B, T, L, kind = c["B"], c["T"], c["L"], c["kind"]
    Hq, Hkv, D = c["Hq"], c["Hkv"], 128
    lens, n_nodes, parents, table, n_blocks = _trees(c, seed)
    s = dict(c=c, M=B * T, status=sd.new_status())
    s["batch"] = sd.Batch(B, T, Hq, Hkv, D, table, lens, n_nodes, parents)
    M, V = s["M"], c["V"]
    i32 = lambda *shape: torch.zeros(shape, dtype=torch.int32, device="cuda")
    f32 = lambda *shape: torch.zeros(shape, dtype=torch.float32, device="cuda")
    if kind != "lmhead":
        s["cache"] = _randn(seed, "cache", (L, 2, n_blocks, Hkv, wl.BLOCK, D))
        s["tree_kv"] = _randn(seed, "tree", (L, 2, B, T, Hkv, D))
        kc, vc = [s["cache"][l, 0] for l in range(L)], [s["cache"][l, 1] for l in range(L)]
        kt, vt = [s["tree_kv"][l, 0] for l in range(L)], [s["tree_kv"][l, 1] for l in range(L)]
        s["layerset"] = sd.LayerSet(kc, vc, kt, vt)
    if kind in ("step", "attention"):
        s["q"] = _randn(seed, "queries", (L, B, T, Hq, D), 2.0)
        s["out"] = torch.zeros((L, B, T, Hq, D), dtype=torch.bfloat16, device="cuda")
        s["att_lse"] = f32(L, B, T, Hq)
        s["per_layer"] = [(sd.kv_layer(kc[l], vc[l]), s["q"][l], kt[l], vt[l], s["out"][l], s["att_lse"][l]) for l in range(L)]
        s["all_layers"] = sd.AttentionLayerSet(kc, vc, list(s["q"]), kt, vt, list(s["out"]), list(s["att_lse"]))
    if kind != "attention":
        _lm_inputs(s, c, seed, parents, n_nodes)
        s["argmax"], s["maxlogit"], s["lse"] = i32(M), f32(M), f32(M)
        s["n_acc"], s["path"], s["out_tok"], s["new_len"] = i32(B), i32(B, T), i32(B, T), i32(B)
    if kind in ("topk", "chain_q", "tree_q"):
        g = _gen(seed, "uniform")
        s["u"], s["w"] = torch.rand((B, T), device="cuda", generator=g), torch.rand((B,), device="cuda", generator=g)
        if kind == "topk":
            s["group_stats"] = f32(*sd.group_stats_shape(M, V))
        else:
            _q_inputs(s, c, seed)
            s["logits"] = f32(M, V)
    s["ws"] = torch.empty(max(256, sd.sd_workspace_bytes(s["batch"], 0 if kind == "attention" else M, 0 if kind == "attention" else V)),
                          dtype=torch.uint8, device="cuda")
    if c["graph"]:
        # a program that replays its step: recorded once, after one direct step
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _issue(s)
        torch.cuda.current_stream().wait_stream(side)
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _issue(s)
    return s


# ---------------------------------------------------------------------------------------------- one pass
def _issue(s):
    c, kind = s["c"], s["c"]["kind"]
    if kind == "draft":
        sd.sd_draft_feature_attention(s["qp"], s["k"], s["v"], c["H"], 1.0 / math.sqrt(128.0), s["out"])
        return
    bt, ws, st = s["batch"], s["ws"], s["status"]
    if kind in ("step", "attention"):
        scale = 1.0 / math.sqrt(128.0)
        sd.sd_tree_prepare(bt, st)
        if c["one_call"]:
            sd.sd_verify_attention_layers(bt, s["all_layers"], scale, ws, st)
        else:
            for cache, q, kt, vt, out, lse in s["per_layer"]:
                sd.sd_verify_attention(bt, cache, q, kt, vt, scale, out, lse, ws, st)
    if kind == "step":
        sd.sd_lmhead_accept_compact(bt, s["hidden"], s["W"], s["draft"], s["layerset"], s["argmax"], s["maxlogit"], s["n_acc"],
                                    s["path"], s["out_tok"], s["new_len"], ws, st)
    elif kind == "lmhead":
        sd.sd_lmhead_argmax(s["hidden"], s["W"], s["argmax"], s["maxlogit"], ws, st)
    elif kind == "topk":
        sd.sd_lmhead_accept_sampled_compact(bt, s["hidden"], s["W"], INV_TEMP, s["draft"], s["u"], s["w"], s["layerset"], s["lse"],
                                            s["group_stats"], s["n_acc"], s["path"], s["out_tok"], s["new_len"], ws, st)
    elif kind in ("chain_q", "tree_q"):
        sd.sd_lmhead_stats_logits(s["hidden"], s["W"], INV_TEMP, None, None, s["lse"], s["logits"], ws, st)
        if kind == "chain_q":
            sd.sd_accept_chain_sampled(bt, s["hidden"], s["W"], INV_TEMP, s["lse"], s["draft"], s["q_tok"], s["q_rows"], s["u"],
                                       s["w"], s["n_acc"], s["path"], s["out_tok"], s["new_len"], ws, st, logits=s["logits"])
        else:
            sd.sd_accept_tree_sampled_q(bt, INV_TEMP, s["lse"], s["logits"], s["draft"], s["q_rows"], s["u"], s["w"], s["n_acc"],
                                        s["path"], s["out_tok"], s["new_len"], st)
        sd.sd_compact_kv(bt, s["layerset"], s["n_acc"], s["path"], st)


def run(state):
    s, kind = state, state["c"]["kind"]
    if "graph" in s:
        s["graph"].replay()
    else:
        _issue(s)
    if kind == "draft":
        return s["out"]
    r = {"status": s["status"]}
    if kind in ("step", "attention"):
        r.update(out=s["out"], att_lse=s["att_lse"])
    if kind in ("step", "lmhead"):
        r.update(argmax=s["argmax"], maxlogit=s["maxlogit"])
    if kind in ("topk", "chain_q", "tree_q"):
        r["lse"] = s["lse"]
        if "logits" in s:
            r["logits"] = s["logits"]
    if kind not in ("attention", "lmhead"):
        r.update(n_acc=s["n_acc"], path=s["path"], out_tok=s["out_tok"], new_len=s["new_len"], cache=s["cache"].view(torch.int16))
    return r


# ---------------------------------------------------------------------------------------------- accounting
def work(case):
    c = case
    if c["kind"] == "draft":
        D = c["H"] * 128
        return {"bytes": c["S"] * c["L"] * D * 2 * (1 if c["same"] else 2) + (c["S"] + 1) * c["Q"] * D * 2,
                "flops": 4.0 * c["S"] * c["L"] * c["Q"] * D}
    B, T, L, kind = c["B"], c["T"], c["L"], c["kind"]
    nodes = B * T * (0.75 if c["ragged_nodes"] else 1.0)
    prefix = (c["prefix_lo"] + c["prefix_hi"]) / 2          # mean length
    bytes_, flops = 0.0, 0.0
    if kind in ("step", "attention"):
        bytes_ += L * (B * prefix * c["Hkv"] * 128 * 4                      # cached K and V, once
                       + nodes * c["Hkv"] * 128 * 4                         # the trees' own
                       + nodes * c["Hq"] * (128 * 2 * 2 + 4))               # q in, out and lse
        flops += L * 4.0 * 128 * c["Hq"] * nodes * (prefix + 1)
    if kind != "attention":
        bytes_ += (c["V"] + B * T) * c["Hd"] * 2.0
        flops += 2.0 * B * T * c["V"] * c["Hd"]
    if kind in ("chain_q", "tree_q"):
        bytes_ += 4.0 * B * T * c["V"] + 2 * 4.0 * B * c["V"]               # logits out; at least the stop row and its q in
    if kind not in ("attention", "lmhead"):
        bytes_ += 2 * 2.0 * L * B * 2 * c["Hkv"] * 128 * 2                  # about two accepted rows read and written
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind in ("step", "attention", "draft"):
        # bf16 outputs, P rounded to bf16; the tokens, lengths and cache bytes must be the same
        return {"rel": 1e-2, "max": 0.1, "differ": 0.0}
    if kind == "lmhead":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}
    # fp32 logits and log-sum-exp; a drawn token may sit on a step of the cumulative distribution
    return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
