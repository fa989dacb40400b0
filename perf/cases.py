"""Cases of the framework's own work: what a training or scoring step over rollout trees calls, over the sizes it meets.

A case names one path (``op``), the shape of its forest and the sizes of its tensors:

  la      scalar-gate linear attention, forward and backward of all rounds (``run_fwd_bwd``)
  score   the same, forward only (reference log-probabilities, the forward of a recomputed layer)
  gk      per-channel-decay linear attention, forward and backward
  attn    attention on compact tokens, forward and backward (MHA and GQA)
  conv    tree-aware causal convolution, forward and backward
  logp    mapped log-probabilities of compact logit rows, forward and backward
  plan    the host side of a step: microbatch plan, and plan and indices of a rank's microbatches

Forests (``shape``), drawn from a seed and cut to exactly ``tokens`` compact tokens:

  agentic  long prompts, turns that fork at their parent's end (fork offsets fall anywhere in a chunk)
  branchy  short segments forking at arbitrary offsets
  replay   a 2k-token root and 16-way fans of branches of 1 to 63 tokens, no fork on a chunk boundary
"""
import math

import numpy as np
import torch

import paper_2608_28158_b200 as hp

DTYPES = {"bf16": torch.bfloat16, "fp32": torch.float32}


# ---------------------------------------------------------------------------------------------------------------- forests
def _agentic_tree(rng, n):
    """A prompt with about 0.65 of the tokens and 9 to 16 turns (lognormal lengths) on at most five levels below it."""
    root = max(1, int(n * rng.uniform(0.55, 0.75)))
    rest = n - root
    m = int(min(rng.integers(9, 17), rest // 32))
    if m < 1:
        return [-1], [0], [n]
    w = np.clip(rng.lognormal(0.0, 1.0, m), 0.1, 8.0)
    lens = np.maximum(16, (w / w.sum() * rest).astype(np.int64))
    lens[np.argmax(lens)] += rest - int(lens.sum())
    par, off, ln, depth, kids = [-1], [0], [root], [0], [0]
    for x in lens.tolist():
        open_ = [i for i in range(len(ln)) if depth[i] < 5 and kids[i] < 4]
        p = int(open_[rng.integers(len(open_))])
        kids[p] += 1
        par.append(p)
        off.append(ln[p])
        ln.append(int(x))
        depth.append(depth[p] + 1)
        kids.append(0)
    return par, off, ln


def _branchy_tree(rng, n):
    """Segments of about 512 tokens (lognormal), up to three children each, forking anywhere inside their parent."""
    par, off, ln, kids, left = [-1], [0], [], [0], n
    while left > 0:
        x = int(np.clip(np.round(rng.lognormal(math.log(512), 0.8)), 16, 4096))
        x = left if left - x < 16 else x
        if ln:
            open_ = [i for i in range(len(ln)) if kids[i] < 3]
            p = int(open_[rng.integers(len(open_))])
            kids[p] += 1
            par.append(p)
            off.append(int(rng.integers(1, ln[p] + 1)))
            kids.append(0)
        ln.append(x)
        left -= x
    return par, off, ln


def _replay_tree(rng, n, root=2048, fanout=16, chunk=64):
    """Two levels of 16-way fans of 1 to 63 tokens; a fork never falls on a chunk boundary if its parent allows it."""
    root = min(root, n)
    par, off, ln, start, left, front = [-1], [0], [root], [0], n - root, [0]
    while left > 0:
        nxt = []
        for v in front:
            for _ in range(fanout):
                if left <= 0:
                    break
                x = min(left, int(rng.integers(1, 64)))
                o = [i for i in rng.integers(1, ln[v] + 1, 8).tolist() if (start[v] + i) % chunk]
                par.append(v)
                off.append(o[0] if o else 1)
                start.append(start[v] + off[-1])
                ln.append(x)
                nxt.append(len(ln) - 1)
                left -= x
        front = nxt
    return par, off, ln


TREES = {"agentic": _agentic_tree, "branchy": _branchy_tree, "replay": _replay_tree}


def forest(shape, tokens, trees, seed):
    """(tree_node_ptr, node_parent, node_fork_off, node_len), int32, of `trees` trees with `tokens` tokens together."""
    rng = np.random.default_rng(seed)
    w = rng.uniform(0.75, 1.25, trees)
    sizes = np.maximum(1, (w / w.sum() * tokens).astype(np.int64))
    sizes[-1] += tokens - int(sizes.sum())
    ptr, par, off, ln = [0], [], [], []
    for n in sizes.tolist():
        p, o, l = TREES[shape](rng, int(n))
        par += p
        off += o
        ln += l
        ptr.append(len(ln))
    return tuple(np.asarray(a, dtype=np.int32) for a in (ptr, par, off, ln))


def case_forest(case):
    return forest(case["shape"], case["tokens"], case["trees"], case["forest"])


def leaf_paths(f):
    """(length of every root-to-leaf trajectory, sum over tokens of their path lengths)."""
    ptr, par, off, ln = (a.tolist() for a in f)
    lens, pairs = [], 0
    for t in range(len(ptr) - 1):
        lo, hi = ptr[t], ptr[t + 1]
        start, tail = [0] * (hi - lo), [False] * (hi - lo)
        for i in range(hi - lo):
            p = par[lo + i]
            if p >= 0:
                start[i] = start[p] + off[lo + i]
                tail[p] = tail[p] or off[lo + i] == ln[lo + p]
            pairs += ln[lo + i] * start[i] + ln[lo + i] * (ln[lo + i] + 1) // 2
        lens += [start[i] + ln[lo + i] for i in range(hi - lo) if not tail[i]]
    return lens, pairs


# ------------------------------------------------------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest call: one small tree, one head, 32-bit (debugging, numerics checks); latency and launches count
        dict(name="la_tiny_fp32", op="la", shape="branchy", tokens=718, trees=1, forest=14, heads=1, d=64, dtype="fp32"),
        # one rollout tree on a head-parallel rank: little work, long chains of chunks
        dict(name="la_small", op="la", shape="branchy", tokens=17695, trees=1, forest=2, heads=4, d=128, dtype="bf16"),
        # a microbatch of agentic trees, 16 heads: the ordinary training call
        dict(name="la_agentic", op="la", shape="agentic", tokens=149270, trees=8, forest=3, heads=16, d=128, dtype="bf16"),
        # a large microbatch, 32 heads
        dict(name="la_large", op="la", shape="agentic", tokens=294449, trees=16, forest=4, heads=32, d=128, dtype="bf16"),
        # thousands of short branches off unaligned forks: replay and state hand-off dominate
        dict(name="la_replay", op="la", shape="replay", tokens=171829, trees=16, forest=5, heads=16, d=128, dtype="bf16"),
        # scoring (no gradients) of one microbatch at the usual 64k-token capacity
        dict(name="la_score", op="score", shape="agentic", tokens=65521, trees=4, forest=6, heads=16, d=128, dtype="bf16"),
        # the per-channel-decay layer on the same kind of microbatch
        dict(name="gk_agentic", op="gk", shape="agentic", tokens=65521, trees=4, forest=6, heads=16, d=128, dtype="bf16"),
        # full-attention layer of a hybrid model on a microbatch, as many key heads as query heads
        dict(name="attn_agentic", op="attn", shape="agentic", tokens=65521, trees=4, forest=6, heads=16, kv_heads=16, d=128, dtype="bf16"),
        # one branchy tree, grouped queries
        dict(name="attn_gqa_small", op="attn", shape="branchy", tokens=9001, trees=1, forest=7, heads=16, kv_heads=4, d=128, dtype="bf16"),
        # the width-4 convolution in front of the linear-attention core
        dict(name="conv_agentic", op="conv", shape="agentic", tokens=149270, trees=8, forest=3, channels=4096, width=4, dtype="bf16"),
        # log-probabilities over a full vocabulary
        dict(name="logp_vocab", op="logp", shape="agentic", tokens=8192, trees=1, forest=8, vocab=157184, dtype="bf16"),
        # host work of one optimizer step: ~1,000 trajectories cut into microbatches, and one rank's first two prepared
        dict(name="plan_step", op="plan", shape="agentic", tokens=2000003, trees=160, forest=9, ranks=4, capacity=65536, own=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, tokens):
    shape = rng.choice(["agentic", "agentic", "branchy", "replay"])
    per_tree = {"agentic": rng.uniform(10000, 20000), "branchy": rng.uniform(8000, 20000), "replay": 10700}[shape]
    return dict(shape=shape, tokens=tokens, trees=max(1, int(math.ceil(tokens / per_tree))), forest=rng.randrange(1 << 20))


def draw(rng):
    op = rng.choice(["la", "la", "la", "la_fp32", "score", "gk", "gk", "attn", "attn", "conv", "logp", "plan"])
    if op == "la_fp32":
        return dict(op="la", **_shape(rng, _log(rng, 300, 12000)), heads=rng.choice([1, 2, 4]), d=64, dtype="fp32")
    if op in ("la", "score", "gk"):
        heads = rng.choice([1, 2, 4, 8, 16, 24, 32])
        most = (2500000 if op == "gk" else 9000000) // heads
        c = _shape(rng, _log(rng, 700, min(most, 290000)))
        if c["shape"] == "replay" and c["tokens"] * heads > 2700000:
            c = dict(c, tokens=2700000 // heads, trees=max(1, 2700000 // heads // 10700))
        return dict(op=op, **c, heads=heads, d=128, dtype="bf16")
    if op == "attn":
        heads, group = rng.choice([4, 8, 16, 32]), rng.choice([1, 1, 2, 4, 8])
        group = min(group, heads)
        return dict(op="attn", **_shape(rng, _log(rng, 1500, 900000 // heads)), heads=heads, kv_heads=heads // group, d=128, dtype="bf16")
    if op == "conv":
        channels = 8 * _log(rng, 64, 768)
        return dict(op="conv", **_shape(rng, _log(rng, 1000, min(600000000 // channels, 290000))), channels=channels, width=4, dtype=rng.choice(["bf16", "bf16", "fp32"]))
    if op == "logp":
        vocab = _log(rng, 16000, 160000)
        return dict(op="logp", **_shape(rng, _log(rng, 500, min(1200000000 // vocab, 16000))), vocab=vocab, dtype=rng.choice(["bf16", "bf16", "fp32"]))
    trees = _log(rng, 16, 160)
    return dict(op="plan", shape="agentic", tokens=trees * rng.randrange(9000, 13000) + rng.randrange(64), trees=trees, forest=rng.randrange(1 << 20), ranks=rng.choice([1, 2, 4]), capacity=65536, own=2)


# ---------------------------------------------------------------------------------------------------------------- prepare
def _dev(a):
    return torch.from_numpy(np.array(a, dtype=np.int32)).cuda()


def _prepare_la(case, f, gen):
    n, H, d, dt = case["tokens"], case["heads"], case["d"], DTYPES[case["dtype"]]
    mk = lambda: torch.randn(n, H, d, generator=gen, device="cuda", dtype=dt)  # noqa: E731
    plan = hp.harts_la_plan(*f).upload()
    s = dict(op=case["op"], plan=plan, q=mk().div_(8.0), k=mk().div_(8.0), v=mk())
    gate = (n, H, d) if case["op"] == "gk" else (n, H)      # log-decays: log(sigmoid(N(3, 1)))
    s["g"] = torch.nn.functional.logsigmoid(torch.randn(gate, generator=gen, device="cuda").add_(3.0))
    s["out"] = {"o": torch.empty_like(s["v"])}
    if case["op"] != "score":
        s["dO"] = mk()
        s["out"].update(dq=torch.empty_like(s["q"]), dk=torch.empty_like(s["k"]), dv=torch.empty_like(s["v"]), dg=torch.empty_like(s["g"]))
    if case["op"] == "gk":
        states, scratch = hp.harts_la_gk_workspace_bytes(plan.tables, H, d, d, hp.HARTS_BF16)
        s["slots"] = torch.empty(max(plan.n_slots, 1) * H * d * d, dtype=torch.float32, device="cuda")
        s["states"] = torch.empty(states, dtype=torch.uint8, device="cuda")
        s["scratch"] = torch.empty(scratch, dtype=torch.uint8, device="cuda")
        s["status"] = torch.zeros(4, dtype=torch.int32, device="cuda")
    else:
        s["ws"] = hp.Workspace(plan, H, d, d, dt)
    return s


def _prepare_attn(case, f, gen):
    n, H, G, d = case["tokens"], case["heads"], case["kv_heads"], case["d"]
    mk = lambda h: torch.randn(n, h, d, generator=gen, device="cuda", dtype=torch.bfloat16)  # noqa: E731
    plan = hp.harts_la_plan(*f)     # rows in the order of the model's linear-attention layers
    s = dict(op="attn", index=hp.harts_attn_index(*f, row_of_token=plan.row_of_token).upload(), scale=1.0 / math.sqrt(d))
    s.update(q=mk(H), k=mk(G), v=mk(G), dO=mk(H))
    s["out"] = dict(o=torch.empty_like(s["q"]), lse=torch.empty(n, H, device="cuda"), dq=torch.empty_like(s["q"]),
                    dk=torch.empty_like(s["k"]), dv=torch.empty_like(s["v"]))
    s["delta"] = torch.empty(n, H, device="cuda")
    s["status"] = torch.zeros(4, dtype=torch.int32, device="cuda")
    return s


def _prepare_conv(case, f, gen):
    n, D, w, dt = case["tokens"], case["channels"], case["width"], DTYPES[case["dtype"]]
    plan = hp.harts_la_plan(*f)
    prev, nxt, cptr, crow = hp.harts_conv_index(*f, row_of_token=plan.row_of_token)
    mk = lambda: torch.randn(n, D, generator=gen, device="cuda", dtype=dt)  # noqa: E731
    s = dict(op="conv", prev=_dev(prev), next=_dev(nxt), cptr=_dev(cptr), crow=_dev(crow), x=mk(), dy=mk())
    s["W"] = torch.randn(D, w, generator=gen, device="cuda").div_(math.sqrt(w))
    s["out"] = dict(y=torch.empty_like(s["x"]), dx=torch.empty_like(s["x"]), dW=torch.empty_like(s["W"]))
    s["scratch"] = torch.empty(hp.harts_conv_scratch_bytes(D, w), dtype=torch.uint8, device="cuda")
    return s


def _prepare_logp(case, f, gen):
    n, V, dt = case["tokens"], case["vocab"], DTYPES[case["dtype"]]
    plan = hp.harts_la_plan(*f)
    # peaked rows: one favoured word stands 6 above N(0, 2^2); half of the tokens are the favoured word of the row before
    fav = torch.randint(0, V, (n,), generator=gen, device="cuda")
    tok = torch.randint(0, V, (n,), generator=gen, device="cuda")
    coin = torch.rand(n, generator=gen, device="cuda") < 0.5
    tok[1:] = torch.where(coin[1:], fav[:-1], tok[1:])
    z = torch.randn(n, V, generator=gen, device="cuda", dtype=dt).mul_(2.0)
    z[torch.arange(n, device="cuda"), fav] += 6.0
    m, y, _ = hp.harts_logp_positions(*f, tok.cpu().numpy(), row_of_token=plan.row_of_token)
    rpp, rp = hp.harts_logp_csr(n, m)
    P = len(m)
    g = torch.randn(P, generator=gen, device="cuda").div_(P)
    g *= torch.rand(P, generator=gen, device="cuda") < 0.6      # the action mask
    out = dict(lse=torch.empty(n, device="cuda"), lam=torch.empty(P, device="cuda"), dz=torch.empty_like(z))
    return dict(op="logp", z=z, m=_dev(m), y=_dev(y), rpp=_dev(rpp), rp=_dev(rp), g=g, out=out,
                status=torch.zeros(4, dtype=torch.int32, device="cuda"))


def prepare(case, seed):
    if case["op"] == "plan":
        f = case_forest(case)       # the trees are the case's, so that tables of every seed have the same sizes; the tokens are the seed's
        ids = np.random.default_rng(seed).integers(0, 157184, case["tokens"], dtype=np.int32)
        base = np.concatenate([[0], np.cumsum(f[3], dtype=np.int64)])
        return dict(op="plan", forest=f, ids=ids, base=base, ranks=case["ranks"], capacity=case["capacity"], own=case["own"])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    f = case_forest(case)
    return {"la": _prepare_la, "score": _prepare_la, "gk": _prepare_la, "attn": _prepare_attn, "conv": _prepare_conv,
            "logp": _prepare_logp}[case["op"]](case, f, gen)


# -------------------------------------------------------------------------------------------------------------------- run
def _run_plan(s):
    mb = hp.harts_mb_plan(*s["forest"], s["ranks"], s["capacity"])
    out = [mb.traj_len, mb.traj_mb, mb.mb_work, mb.mb_replica, mb.mb_slot]
    mine = [int(i) for i in np.flatnonzero(mb.mb_replica == 0)]
    for i in sorted(mine, key=lambda i: int(mb.mb_slot[i]))[:s["own"]]:
        ptr, par, off, ln, src = mb.extract(i)
        f = (ptr, par, off, ln)
        plan = hp.harts_la_plan(*f).upload()
        attn = hp.harts_attn_index(*f, row_of_token=plan.row_of_token).upload()
        conv = hp.harts_conv_index(*f, row_of_token=plan.row_of_token)
        ids = np.concatenate([s["ids"][s["base"][j]:s["base"][j] + n] for j, n in zip(src.tolist(), ln.tolist())])
        m, y, tp = hp.harts_logp_positions(*f, ids, row_of_token=plan.row_of_token)
        rpp, rp = hp.harts_logp_csr(plan.n_rows, m)
        out += [src, plan.row_of_token, plan.seq_own_begin, plan.seq_init_slot, plan.replay_row, plan.slot_chunk, plan.rg_entry,
                plan.seq_order, plan.blob.view(torch.int32), attn.dev, *conv, m, y, tp, rpp, rp]
    return out


def run(s):
    op = s["op"]
    if op == "plan":
        return _run_plan(s)
    o = s["out"]
    if op == "la":
        return hp.run_fwd_bwd(s["plan"], s["ws"], s["q"], s["k"], s["v"], s["g"], s["dO"], out=o)
    if op == "score":
        return hp.run_fwd_bwd(s["plan"], s["ws"], s["q"], s["k"], s["v"], s["g"], None, out=o, backward=False)
    if op == "gk":
        hp.harts_la_gk_fwd(s["plan"], 0, s["q"], s["k"], s["v"], s["g"], o["o"], s["slots"], s["states"], 0, s["status"])
        hp.harts_la_gk_bwd(s["plan"], 0, s["q"], s["k"], s["v"], s["g"], s["dO"], o["dq"], o["dk"], o["dv"], o["dg"], s["states"],
                           s["scratch"], 0, s["status"])
    elif op == "attn":
        hp.harts_attn_fwd(s["index"], s["q"], s["k"], s["v"], o["o"], o["lse"], s["scale"], s["status"])
        hp.harts_attn_bwd(s["index"], s["q"], s["k"], s["v"], o["o"], o["lse"], s["dO"], o["dq"], o["dk"], o["dv"], s["delta"],
                          s["scale"], s["status"])
    elif op == "conv":
        hp.harts_conv_fwd(s["x"], s["W"], s["prev"], o["y"])
        hp.harts_conv_bwd(s["x"], s["W"], s["dy"], s["next"], s["cptr"], s["crow"], o["dx"], o["dW"], s["scratch"])
    else:
        hp.harts_logp_fwd(s["z"], s["m"], s["y"], o["lse"], o["lam"], dev_status=s["status"])
        hp.harts_logp_bwd(s["z"], s["y"], s["rpp"], s["rp"], o["lse"], s["g"], o["dz"], dev_status=s["status"])
    return o


# ------------------------------------------------------------------------------------------------------- work, tolerance
def work(case):
    op, n = case["op"], case["tokens"]
    e = 4 if case.get("dtype") == "fp32" else 2
    if op in ("la", "score", "gk"):
        H, d, gate = case["heads"], case["d"], 4 * (case["d"] if case["op"] == "gk" else 1)
        fwd, bwd = 4 * 64 * d + 4 * d * d, 5 * 2 * 64 * d + 4 * 2 * d * d       # per token and head, chunks of 64
        if op == "score":
            return {"bytes": n * H * (4 * d * e + gate), "flops": n * H * fwd}
        return {"bytes": n * H * (9 * d * e + 2 * gate), "flops": n * H * (fwd + bwd)}
    if op == "attn":
        H, G, d = case["heads"], case["kv_heads"], case["d"]
        pairs = leaf_paths(case_forest(case))[1]
        return {"bytes": n * (4 * H * d * e + 4 * G * d * e + 4 * H), "flops": 14 * d * H * pairs}
    if op == "conv":
        return {"bytes": 4 * n * case["channels"] * e, "flops": 3 * 2 * n * case["channels"] * case["width"]}
    if op == "logp":
        return {"bytes": 2 * n * case["vocab"] * e, "flops": 8 * n * case["vocab"]}
    own = min(n, case["own"] * case["capacity"])        # one rank's microbatches: about 30 words of tables for each token
    return {"bytes": 120 * own, "flops": 0}


def tolerance(case):
    if case["op"] == "plan":
        return "exact"
    if case["dtype"] == "fp32":
        return {"rel": 1e-5}
    return {"rel": 1e-2 if case["op"] in ("la", "score", "gk", "attn") else 4e-3}
