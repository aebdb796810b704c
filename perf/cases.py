"""Timed cases of the speculative-decoding hot path, through the binding that users call.

Five kinds of work, each one a part of serving a long-video request:

  decode  one draft step: attention of one new query token per sequence over the draft's K/V cache
  step    one verification of a drafted chain: append the window's K/V, attention of its gamma + 1
          queries over the target's cache, greedy acceptance, rollback of the rejected rows
  tree    one verification of a drafted tree: attention of its nodes, acceptance along the tree
  rate    the rating of the video tokens from the target's language-to-video attention (once per
          request), with or without the log-sum-exps that the target's prefill may have left
  prune   two-stage selection of the kept video tokens and the gather of their K/V rows into the
          draft's cache (once per request)

A call covers ``layers`` layers: all of them where a program batches a model's layers, one where it
calls the path from each layer of a forward pass.  Sequences of a batch are ragged: their lengths
follow from ``tokens`` and the batch index.  Head shapes, lengths and grids are those of the five
workloads in ``synth.workload`` and of the tests.
"""
import math

import torch

from paper_2508_16201_b200 import specvlm

DRAFT_HEADS = ((28, 4, 128), (4, 1, 64))                    # (query heads, KV heads, head_dim)
TARGET_HEADS = ((64, 8, 128), (40, 8, 128), (28, 4, 128), (8, 2, 64))
PAGE = 64


def listed():
    return [
        # a draft layer's decode call on the pruned cache of a 32-frame video: the smallest call of a
        # program that runs its model layer by layer
        dict(name="decode-layer", kind="decode", layers=1, q_heads=28, kv_heads=4, head_dim=128, batch=1, tokens=755,
             paged=False),
        # the draft step of the 32-frame workload: all 28 layers, 10 % of the video tokens + the text
        dict(name="decode-pruned", kind="decode", layers=28, q_heads=28, kv_heads=4, head_dim=128, batch=1, tokens=755,
             paged=False),
        # batched serving: 16 ragged pruned caches of up to 128 frames in 64-token pages
        dict(name="decode-batch", kind="decode", layers=28, q_heads=28, kv_heads=4, head_dim=128, batch=16, tokens=2700,
             paged=True),
        # one target layer verifying a chain of 5 drafts over a 32-frame video
        dict(name="step-layer", kind="step", layers=1, q_heads=64, kv_heads=8, head_dim=128, batch=1, tokens=6400, gamma=5,
             vocab=152064, paged=False),
        # the same for all 80 layers in one call: the headline verification
        dict(name="step-80-layers", kind="step", layers=80, q_heads=64, kv_heads=8, head_dim=128, batch=1, tokens=6400,
             gamma=5, vocab=152064, paged=False),
        # batched serving with a long window: 4 ragged videos of up to 128 frames, paged, gamma = 8 (72 query rows
        # per KV head); 40 layers
        dict(name="step-batch", kind="step", layers=40, q_heads=64, kv_heads=8, head_dim=128, batch=4, tokens=25216,
             gamma=8, vocab=152064, paged=True),
        # tree drafting, the default of the method: 26 nodes (208 query rows per KV head) over the 32-frame video
        dict(name="tree-26", kind="tree", layers=80, q_heads=64, kv_heads=8, head_dim=128, batch=1, tokens=6400, nodes=26,
             vocab=152064, paged=False),
        # the tiny workload: 4 frames, 64 text tokens, one layer, head_dim 64
        dict(name="rate-tiny", kind="rate", layers=1, q_heads=8, kv_heads=2, head_dim=64, batch=1, video=784, text=64,
             lse=False, paged=False),
        # rating of a 32-frame video after a prefill that kept its log-sum-exps
        dict(name="rate-80-layers", kind="rate", layers=80, q_heads=64, kv_heads=8, head_dim=128, batch=1, video=6272,
             text=128, lse=True, paged=False),
        # rating on the 20 x 36 grid, 32 temporal groups, 5 query heads per KV head, from the queries alone
        dict(name="rate-64-layers", kind="rate", layers=64, q_heads=40, kv_heads=8, head_dim=128, batch=1, video=23040,
             text=256, lse=False, paged=False),
        # selection + gather of a 32-frame video: fixed Stage-I count, 10 % kept
        dict(name="prune-32-frames", kind="prune", layers=28, kv_heads=4, head_dim=128, batch=1, frames=32, grid=196,
             text=128, permille=100, lambda_permille=-1, paged=False),
        # the same for 256 frames with the cumulative-score rule (lambda 0.4)
        dict(name="prune-256-frames", kind="prune", layers=28, kv_heads=4, head_dim=128, batch=1, frames=256, grid=196,
             text=128, permille=100, lambda_permille=400, paged=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("decode", "decode", "step", "step", "tree", "rate", "rate", "prune", "prune"))
    paged = rng.random() < 0.5
    while True:
        if kind == "decode":
            hq, hkv, d = rng.choice(DRAFT_HEADS)
            c = dict(kind=kind, layers=_log(rng, 1, 28), q_heads=hq, kv_heads=hkv, head_dim=d, batch=_log(rng, 1, 16),
                     tokens=_log(rng, 40, 50000), paged=paged)
            cost = work(c)["bytes"] / 8e9
        elif kind == "step":
            hq, hkv, d = rng.choice(TARGET_HEADS)
            c = dict(kind=kind, layers=_log(rng, 1, 80), q_heads=hq, kv_heads=hkv, head_dim=d, batch=_log(rng, 1, 8),
                     tokens=_log(rng, 200, 50000), gamma=rng.randint(1, 8), vocab=_log(rng, 1024, 152064), paged=paged)
            cost = work(c)["bytes"] / 8e9
        elif kind == "tree":
            hq, hkv, d = rng.choice(TARGET_HEADS)
            c = dict(kind=kind, layers=_log(rng, 1, 80), q_heads=hq, kv_heads=hkv, head_dim=d, batch=_log(rng, 1, 4),
                     tokens=_log(rng, 200, 25000), nodes=rng.randint(5, 40), vocab=_log(rng, 1024, 152064), paged=paged)
            cost = max(work(c)["bytes"] / 4e9, work(c)["flops"] / 2e12)
        elif kind == "rate":
            hq, hkv, d = rng.choice(TARGET_HEADS)
            c = dict(kind=kind, layers=_log(rng, 1, 80), q_heads=hq, kv_heads=hkv, head_dim=d, batch=_log(rng, 1, 4),
                     video=_log(rng, 196, 50176), text=rng.randint(16, 256), lse=rng.random() < 0.5, paged=paged)
            cost = work(c)["flops"] / 4e12
        else:
            d = rng.choice((128, 128, 64))
            c = dict(kind=kind, layers=_log(rng, 1, 28), kv_heads=4 if d == 128 else 1, head_dim=d, batch=_log(rng, 1, 16),
                     frames=_log(rng, 4, 256), grid=rng.choice((196, 720, 169)), text=rng.randint(16, 256),
                     permille=_log(rng, 50, 500), lambda_permille=rng.choice((-1, 400, 500)), paged=paged)
            cost = 1.0 if c["frames"] * c["grid"] <= 57344 else 2.0
            src = c["layers"] * c["kv_heads"] * d * 4 * c["batch"] * c["frames"] * c["grid"]
            cost = max(cost, src / 16e9)
        if cost <= 1.0:
            return c


# ------------------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _randn(shape, g):
    t = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
    for layer in t:
        layer.normal_(generator=g)
    return t


def _ragged(n, batch):
    """Lengths of a batch: quarters of n, a few tokens apart so that most end inside a tile."""
    return [max(1, n * (4 - b % 4) // 4 - 13 * b % 29 * (b > 0)) for b in range(batch)]


def _cache(c, lens, room, g, fill=True):
    """A K/V cache for sequences of ``lens`` tokens with space for ``room`` more each; paged caches
    take scattered pages of a pool."""
    caps = [n + room for n in lens]
    table = None
    if c["paged"]:
        need = [-(-n // PAGE) for n in caps]
        shape = (c["layers"], sum(need) + 3, c["kv_heads"], PAGE, c["head_dim"])
        perm = torch.randperm(shape[1], generator=g, device="cuda", dtype=torch.int32)
        table = torch.full((len(lens), max(need)), -1, dtype=torch.int32, device="cuda")
        at = 0
        for b, n in enumerate(need):
            table[b, :n] = perm[at:at + n]
            at += n
    else:
        shape = (c["layers"], len(lens), c["kv_heads"], max(caps), c["head_dim"])
    if fill:
        k, v = _randn(shape, g), _randn(shape, g)
    else:
        k, v = (torch.zeros(shape, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    seq = torch.tensor(lens, dtype=torch.int32, device="cuda")
    return specvlm.KvCache(k, v, seq, max(caps), table)


def _rows(t, cache, layer, b, n):
    """The first n token rows of sequence b in one layer: [kv_heads][n][head_dim]."""
    if cache.block_table is None:
        return t[layer, b, :, :n]
    blocks = cache.block_table[b, :-(-n // PAGE)].long()
    return t[layer, blocks].transpose(0, 1).reshape(t.shape[2], -1, t.shape[4])[:, :n]


def _logits(batch, rows, vocab, g):
    """fp32 target logits, and draft tokens that equal the row's choice about two times in three."""
    x = torch.empty((batch, rows, vocab), dtype=torch.float32, device="cuda").normal_(generator=g)
    hit = torch.rand((batch, rows), generator=g, device="cuda") < 0.66
    other = torch.randint(0, vocab, (batch, rows), generator=g, device="cuda")
    return x, torch.where(hit, x.argmax(-1), other).to(torch.int32)


def _parents(batch, nodes):
    """A tree of falling width, as static draft trees are: the first nodes have more children."""
    return torch.tensor([[-1] + [(t - 1) // 3 if t < nodes // 2 else t // 2 for t in range(1, nodes)]] * batch,
                        dtype=torch.int32, device="cuda")


def _tree_tokens(top, parents, g, vocab):
    """Node tokens [batch][nodes]: a child carries its parent's target choice two times in five."""
    par = parents.clamp_min(0).long()
    hit = torch.rand(parents.shape, generator=g, device="cuda") < 0.4
    other = torch.randint(0, vocab, parents.shape, generator=g, device="cuda")
    return torch.where(hit, top.gather(1, par), other).to(torch.int32)


def _salient(c, cache, q, lens, g):
    """5 % of the video tokens lean towards the text queries, as in the benchmark's inputs."""
    group = c["q_heads"] // c["kv_heads"]
    at = 0
    for b, nv in enumerate(lens):
        nt = c["text"]
        u = q[:, at:at + nt].float().view(c["layers"], nt, c["kv_heads"], group, c["head_dim"]).mean((1, 3))
        u = (2.0 * u / u.norm(dim=-1, keepdim=True)).unsqueeze(2)
        at += nt
        idx = torch.randperm(nv, generator=g, device="cuda")[:max(1, nv // 20)]
        blk, off = (cache.block_table[b, idx // PAGE].long(), idx % PAGE) if c["paged"] else (torch.full_like(idx, b), idx)
        for layer in range(c["layers"]):
            k = cache.k[layer]
            k[blk, :, off] = (k[blk, :, off].float() + u[layer].transpose(0, 1)).to(torch.bfloat16)


def _text_logits(c, s, layer, b, n, dtype):
    """Scaled causal logits of sequence b's text queries in one layer: per KV head [text * group][n]."""
    nt, group, d = c["text"], c["q_heads"] // c["kv_heads"], c["head_dim"]
    q = s["q"][layer, b * nt:(b + 1) * nt].view(nt, c["kv_heads"], group, d).to(dtype)
    hidden = torch.arange(n, device="cuda") > (n - nt + torch.arange(nt, device="cuda")).repeat_interleave(group)[:, None]
    k = _rows(s["cache"].k, s["cache"], layer, b, n).to(dtype)
    for h in range(c["kv_heads"]):
        x = (q[:, h].reshape(-1, d) @ k[h].T).mul_(s["scale"])
        yield h, x.masked_fill_(hidden, float("-inf"))


def _row_lse(c, s, dtype=torch.float32):
    nt, group = c["text"], c["q_heads"] // c["kv_heads"]
    lse = torch.empty((c["layers"], nt * c["batch"], c["kv_heads"], group), dtype=dtype, device="cuda")
    for layer in range(c["layers"]):
        for b, nv in enumerate(s["video_len"]):
            for h, x in _text_logits(c, s, layer, b, nv + nt, dtype):
                lse[layer, b * nt:(b + 1) * nt, h] = torch.logsumexp(x, -1).view(nt, group)
    return lse.view(c["layers"], nt * c["batch"], c["q_heads"])


def _cu(lens):
    cu = [0]
    for n in lens:
        cu.append(cu[-1] + n)
    return cu


def prepare(case, seed):
    c, g = case, _gen(seed)
    s = dict(case=c)
    if c["kind"] != "prune":
        s["scale"] = 1.0 / math.sqrt(c["head_dim"])
    L, B = c["layers"], c["batch"]
    if c["kind"] == "decode":
        s["cache"] = _cache(c, _ragged(c["tokens"], B), 0, g)
        s["q"] = _randn((L, B, c["q_heads"], c["head_dim"]), g)
        s["out"] = torch.empty_like(s["q"])
        nbytes = specvlm.attn_workspace_bytes(s["cache"], B, c["q_heads"], 0)
        s["ws"] = torch.empty(max(nbytes, 256), dtype=torch.uint8, device="cuda")
    elif c["kind"] == "step":
        n = c["gamma"] + 1
        s["cache"] = _cache(c, _ragged(c["tokens"], B), n, g)
        s["lens"] = s["cache"].seq_lens.clone()
        s["new_k"], s["new_v"] = (_randn((L, B, n, c["kv_heads"], c["head_dim"]), g) for _ in range(2))
        s["q"] = _randn((L, B, n, c["q_heads"], c["head_dim"]), g)
        s["out"] = torch.empty_like(s["q"])
        s["logits"], drafts = _logits(B, n, c["vocab"], g)
        s["drafts"] = drafts[:, :-1].contiguous()
        nbytes = specvlm.attn_workspace_bytes(s["cache"], B, c["q_heads"], c["gamma"])
        s["ws"] = torch.empty(max(nbytes, 256), dtype=torch.uint8, device="cuda")
        s["accept_ws"] = torch.empty(specvlm.accept_workspace_bytes(B, c["gamma"], c["vocab"]), dtype=torch.uint8, device="cuda")
        s["accept"] = tuple(torch.empty(shape, dtype=torch.int32, device="cuda") for shape in ((B,), (B,), (B, n)))
    elif c["kind"] == "tree":
        n = c["nodes"]
        s["cache"] = _cache(c, [x + n for x in _ragged(c["tokens"], B)], 0, g)
        s["q"] = _randn((L, B, n, c["q_heads"], c["head_dim"]), g)
        s["out"] = torch.empty_like(s["q"])
        s["parents"] = _parents(B, n)
        s["logits"], _ = _logits(B, n, c["vocab"], g)
        s["tokens"] = _tree_tokens(s["logits"].argmax(-1), s["parents"], g, c["vocab"])
        s["accept"] = specvlm.accept_tree_buffers(B, n, c["vocab"], "cuda", want_argmax=True)
    elif c["kind"] == "rate":
        s["video_len"] = _ragged(c["video"], B)
        s["text_cu"] = _cu([c["text"]] * B)
        s["cache"] = _cache(c, [n + c["text"] for n in s["video_len"]], 0, g)
        s["q"] = _randn((L, s["text_cu"][-1], c["q_heads"], c["head_dim"]), g)
        _salient(c, s["cache"], s["q"], s["video_len"], g)
        s["video_cu"] = _cu(s["video_len"])
        s["row_lse"] = _row_lse(c, s) if c["lse"] else None
        s["scores"] = torch.empty(s["video_cu"][-1], dtype=torch.float32, device="cuda")
        nbytes = specvlm.stage1_scores_workspace_bytes(s["cache"], s["text_cu"], s["video_len"], c["q_heads"])
        s["ws"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    else:
        s["n_frames"] = [max(1, c["frames"] * (4 - b % 4) // 4) for b in range(B)]
        s["video_len"] = [f * c["grid"] for f in s["n_frames"]]
        s["k_total"] = [n * c["permille"] // 1000 for n in s["video_len"]]
        s["video_cu"], s["kept_cu"] = _cu(s["video_len"]), _cu(s["k_total"])
        s["src_len"] = [n + c["text"] for n in s["video_len"]]
        s["src"] = _cache(c, s["src_len"], 0, g)
        s["dst"] = _cache(c, [k + c["text"] for k in s["k_total"]], 0, g, fill=False)
        # mean attention probabilities: a near-uniform bulk and 5 % salient tokens
        x = torch.empty(s["video_cu"][-1], dtype=torch.float32, device="cuda").normal_(generator=g).mul_(0.4).exp_()
        x *= 1.0 + 4.0 * (torch.rand(x.shape, generator=g, device="cuda") < 0.05)
        s["scores"] = torch.cat([0.95 * p / p.sum() for p in x.split(s["video_len"])])
        s["kept"] = torch.empty(max(1, s["kept_cu"][-1]), dtype=torch.int32, device="cuda")
        s["k_stage1"] = torch.empty(B, dtype=torch.int32, device="cuda")
    return s


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "decode":
        return specvlm.draft_decode_attn(s["cache"], s["q"], s["scale"], out=s["out"], ws=s["ws"])
    if c["kind"] == "step":
        cache = s["cache"]
        cache.seq_lens.copy_(s["lens"])                     # the step starts from the same sequences again
        specvlm.append_kv(cache, s["new_k"], s["new_v"])
        out = specvlm.verify_attn(cache, s["q"], c["gamma"], s["scale"], out=s["out"], ws=s["ws"])
        n, token, choice = specvlm.accept(s["logits"], s["drafts"], ws=s["accept_ws"], out=s["accept"])
        specvlm.rollback_kv(cache.seq_lens, n, c["gamma"])
        return dict(out=out, n=n, token=token, choice=choice, lens=cache.seq_lens, k=cache.k, v=cache.v)
    if c["kind"] == "tree":
        out = specvlm.verify_tree_attn(s["cache"], s["q"], s["parents"], s["scale"], out=s["out"])
        n, token, path, choice = specvlm.accept_tree(s["logits"], s["tokens"], s["parents"], out=s["accept"])
        return dict(out=out, n=n, token=token, path=path, choice=choice)
    if c["kind"] == "rate":
        zeros = [0] * c["batch"]
        return specvlm.stage1_scores(s["cache"], s["q"], s["text_cu"], s["video_len"], zeros, s["video_len"], s["video_cu"],
                                     s["scale"], scores=s["scores"], ws=s["ws"], row_lse=s["row_lse"])
    k1 = None
    if c["lambda_permille"] < 0:
        kept = specvlm.select(s["scores"], s["video_cu"], s["n_frames"], c["grid"], [k // 2 for k in s["k_total"]],
                              s["k_total"], s["kept_cu"], kept_idx=s["kept"])
    else:
        kept, k1 = specvlm.select_top_p(s["scores"], s["video_cu"], s["n_frames"], c["grid"],
                                        [c["lambda_permille"]] * c["batch"], s["k_total"], s["kept_cu"],
                                        kept_idx=s["kept"], k_stage1_out=s["k_stage1"])
    specvlm.gather_kv(s["src"], kept, s["kept_cu"], [0] * c["batch"], s["video_len"], s["src_len"], s["dst"])
    return dict(kept=kept, k1=k1, k=s["dst"].k, v=s["dst"].v)


# ------------------------------------------------------------------------------------------ accounting
def work(case):
    """K and V rows of every cached token once, queries and outputs once, logits once; two flops per
    multiply-add of the products QK^T and PV (the rating needs QK^T alone)."""
    c, L = case, case["layers"]
    row = c["kv_heads"] * c["head_dim"] * 2                 # bytes of a token's K (or V) in one layer
    if c["kind"] == "prune":
        frames = [max(1, c["frames"] * (4 - b % 4) // 4) for b in range(c["batch"])]
        kept = sum(f * c["grid"] * c["permille"] // 1000 + c["text"] for f in frames)
        return {"bytes": 4 * L * kept * row + 4 * sum(frames) * c["grid"], "flops": 0}
    qrow = c["q_heads"] * c["head_dim"]
    if c["kind"] == "rate":
        video = _ragged(c["video"], c["batch"])
        text = c["text"] * c["batch"]
        return {"bytes": L * (sum(video) + text) * row + L * text * (qrow * 2 + 4 * c["q_heads"] * c["lse"]) + 4 * sum(video),
                "flops": sum(2 * L * c["text"] * qrow * (n + c["text"]) for n in video)}
    n_q = {"decode": 1, "step": c.get("gamma", 0) + 1, "tree": c.get("nodes", 0)}[c["kind"]]
    keys = sum(_ragged(c["tokens"], c["batch"])) + (n_q * c["batch"] if n_q > 1 else 0)
    nbytes = 2 * L * keys * row + 4 * L * c["batch"] * n_q * qrow
    if c["kind"] == "step":
        nbytes += 4 * L * c["batch"] * n_q * row            # the new rows, read and written
    if n_q > 1:
        nbytes += 4 * c["batch"] * n_q * c["vocab"]
    return {"bytes": nbytes, "flops": 4 * L * n_q * qrow * keys}


def tolerance(case):
    if case["kind"] == "prune":
        return "exact"
    if case["kind"] == "rate":
        # fp32 products and sums, exponentials good to a few 1e-6 each: 1e-7 to 6e-7 against 64 bits
        return {"rel": 4e-6, "max": 4e-5}
    # probabilities and outputs in bf16 (2.3e-3 against 64 bits); accepted tokens and cache rows are exact
    return {"rel": 1e-2, "max": 0.1, "differ": 0.0}


def exact(case, seed):
    """The same outputs in 64 bits, from plain tensor operations."""
    c = case
    if c["kind"] == "prune":
        return None
    s = prepare(c, seed)
    if c["kind"] == "rate":
        lse = s["row_lse"].double() if c["lse"] else None
        nt, group = c["text"], c["q_heads"] // c["kv_heads"]
        total = torch.zeros(s["video_cu"][-1], dtype=torch.float64, device="cuda")
        for layer in range(c["layers"]):
            for b, nv in enumerate(s["video_len"]):
                for h, x in _text_logits(c, s, layer, b, nv + nt, torch.float64):
                    if lse is None:
                        p = torch.softmax(x, -1)
                    else:
                        p = (x - lse[layer, b * nt:(b + 1) * nt].view(nt, c["kv_heads"], group)[:, h].reshape(-1, 1)).exp_()
                    total[s["video_cu"][b]:s["video_cu"][b + 1]] += p[:, :nv].sum(0)
        return total / (c["layers"] * c["q_heads"] * nt)
    cache, group, d = s["cache"], c["q_heads"] // c["kv_heads"], c["head_dim"]
    q = s["q"].unsqueeze(2) if c["kind"] == "decode" else s["q"]
    n_q = q.shape[2]
    if c["kind"] == "step":
        before = [int(n) for n in s["lens"]]
        for b, n in enumerate(before):                # the window's rows take their places
            for t in range(n_q):
                at = (cache.block_table[b, (n + t) // PAGE].long(), (n + t) % PAGE) if c["paged"] else (b, n + t)
                cache.k[:, at[0], :, at[1]] = s["new_k"][:, b, t]
                cache.v[:, at[0], :, at[1]] = s["new_v"][:, b, t]
        lens = [n + n_q for n in before]
    else:
        lens = [int(n) for n in cache.seq_lens]
    window = torch.ones((n_q, n_q), dtype=torch.bool, device="cuda").tril()
    if c["kind"] == "tree":
        parents = s["parents"][0].tolist()
        window = torch.zeros((n_q, n_q), dtype=torch.bool, device="cuda")
        for t in range(n_q):
            a = t
            while a >= 0:
                window[t, a] = True
                a = parents[a]
    window = window.repeat_interleave(group, 0)
    out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
    for layer in range(c["layers"]):
        for b, n in enumerate(lens):
            k, v = (_rows(t, cache, layer, b, n).double() for t in (cache.k, cache.v))
            x = q[layer, b].double().view(n_q, c["kv_heads"], group, d).transpose(0, 1).reshape(c["kv_heads"], n_q * group, d)
            x = (x @ k.transpose(1, 2)).mul_(s["scale"])
            x[:, :, n - n_q:].masked_fill_(~window, float("-inf"))
            o = torch.softmax(x, -1) @ v
            out[layer, b] = o.view(c["kv_heads"], n_q, group, d).transpose(0, 1).reshape(n_q, c["q_heads"], d)
    if c["kind"] == "decode":
        return out.squeeze(2)
    return dict(out=out)
