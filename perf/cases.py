"""The calls that a user of libc2t makes, as measurable cases: whole decode steps from the smallest (one sequence, a
32000-token vocabulary) to the largest (64 sequences, 128256 tokens), both logits types, the truncated entropy, the two
acceptance walks, a step fed from host memory, one rank's share of a vocabulary-parallel step, and the two calls that
stand alone (row arg-max without a workspace, dense attention mask).

A case is a dict of plain values; `prepare` makes what a serving loop holds before the call (a context, its logits on
the GPU or in pinned host memory), `run` makes the calls of one pass, `work` states the bytes and operations the pass
cannot do without.  Logits are the seeded Gumbel + Zipf rows of `c2t_inputs`; the target rows are changed so that
their arg-maxes follow a path of the final tree over a few levels, as they do when a trained draft model is in use
(the synthetic rows alone accept next to nothing).
"""
import torch

import c2t_inputs
import paper_2502_13652_b200 as c2t
from paper_2502_13652_b200.vocab_parallel import shard_ranges

ACCEPT_LEVELS = (2, 5)       # accepted draft tokens per step that the target rows are made to give, at most


def _step(name, kind="step", **kw):
    """A decode step: kind "step" (all-rows acceptance), "lazy" (rows on the path only), "host" (pinned host buffers)
    or "shard" (one rank of a vocabulary-parallel group, `shards` ranks)."""
    c = dict(kind=kind, batch=1, vocab=32000, dtype="bf16", depth=8, topk=10, frontier=10, budget=60, threshold=0.5,
             classifier="mlp", hidden=16, top_m=0, add_all=False, scale=4.0, shards=1)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one interactive user, 32000-token vocabulary, fp32 logits: the smallest step, nothing but latency
        _step("step_b1_v32000_f32", batch=1, vocab=32000, dtype="f32", depth=6),
        # one interactive user, 128256-token vocabulary, the deep and wide single-sequence tree
        _step("step_b1_v128256_bf16", batch=1, vocab=128256, depth=10, topk=8, frontier=16, budget=80),
        # a handful of users on one GPU: the ordinary step
        _step("step_b8_v32000_bf16", batch=8, vocab=32000),
        # the throughput step: a full batch, the largest vocabulary
        _step("step_b64_v128256_bf16", batch=64, vocab=128256),
        # a draft head that leaves its logits in fp32
        _step("step_b32_v128256_f32", batch=32, vocab=128256, dtype="f32", budget=40),
        # the entropy feature over the 1000 most probable tokens, as the paper trains its classifier
        _step("step_top1000_b16_v128256_bf16", batch=16, vocab=128256, depth=6, top_m=1000),
        # expand + rerank by joint probability over all survivors, an odd batch and a vocabulary with added tokens
        _step("step_joint_b5_v32003_f32", batch=5, vocab=32003, dtype="f32", depth=6, threshold=0.0,
              classifier="joint", add_all=True, scale=1.0),
        # the throughput step with the acceptance walk that reads only the rows on the accepted path
        _step("lazy_b64_v128256_bf16", kind="lazy", batch=64, vocab=128256),
        # draft and target models on another device: the step's logits come from pinned host memory
        _step("host_b8_v32000_bf16", kind="host", batch=8, vocab=32000),
        # one rank of an 8-way vocabulary-parallel group: its token range of every row, the others' records at hand
        _step("shard8_b64_v128256_bf16", kind="shard", batch=64, vocab=128256, shards=8),
        # greedy tokens of a plain decoding batch, for a caller that may not allocate
        dict(name="argmax_r256_v128256_bf16", kind="argmax", rows=256, vocab=128256, dtype="bf16"),
        # the additive attention mask of a batch for an attention kernel without bit masks
        dict(_step("mask_b64_kv4160_bf16", kind="mask", batch=64, vocab=4096, depth=6), kv_len=4160, prefix=4096,
             out="bf16"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["step"] * 5 + ["lazy"] * 2 + ["top_m", "host", "shard", "argmax", "mask"])
    dtype = rng.choice(["bf16", "bf16", "f32"])
    vocab = rng.choice([32000, 128256, _log_uniform(rng, 4000, 150000)])
    if kind == "argmax":
        rows = _log_uniform(rng, 1, 4096)
        esz = 2 if dtype == "bf16" else 4
        while rows * vocab * esz > 1e9:
            rows = rows * 2 // 3
        return dict(kind="argmax", rows=rows, vocab=vocab, dtype=dtype)
    mlp = rng.random() < 0.7
    frontier = rng.choice([10, 10, rng.randint(3, 24)])
    c = _step(None, kind="step" if kind == "top_m" else kind, batch=_log_uniform(rng, 1, 96), vocab=vocab, dtype=dtype,
              depth=rng.randint(4, 10), topk=rng.choice([10, 10, rng.randint(3, 16)]), frontier=frontier,
              budget=rng.choice([20, 40, 60, 80]), threshold=rng.choice([0.3, 0.5]) if mlp else rng.choice([0.0, 1e-3]),
              classifier="mlp" if mlp else "joint", add_all=not mlp and rng.random() < 0.5,
              scale=rng.choice([1.0, 4.0, 4.0, 8.0]))
    if kind == "top_m":
        c["top_m"] = rng.choice([1000, rng.randint(200, 1500)])
    if kind == "shard":
        c["shards"] = rng.choice([2, 4, 8])
    if kind == "host":
        c["vocab"] = -(-vocab // 8) * 8              # the host buffers are contiguous: rows of whole 16 bytes
    if kind == "mask":
        c.update(vocab=4096, kv_len=_log_uniform(rng, 256, 8192), out=rng.choice(["bf16", "f32"]))
        c["prefix"] = c["kv_len"] - rng.randint(0, 80)
    most = {"host": 1e8, "shard": 3e8, "mask": 2e8}.get(kind, 7e8 if kind == "top_m" else 2.1e9)
    while c["batch"] > 1 and work(c)["bytes"] * (c["shards"] if kind == "shard" else 1) > most:
        c["batch"] = c["batch"] * 2 // 3
    while work(c)["bytes"] > most and c["depth"] > 2:
        c["depth"] -= 1
    return c


# ---------------------------------------------------------------------------- what a pass cannot do without

def _rows_per_level(c):
    """Frontier rows per sequence and level when the threshold drops nothing (it does not at these settings, except for
    the joint classifier at a positive one)."""
    rows, n = [], 1
    for _ in range(c["depth"]):
        rows.append(n)
        n = min(c["frontier"], n * c["topk"])
    return rows


def _final_nodes(c):
    rows = _rows_per_level(c)
    grown = sum(r * c["topk"] for r in rows) if c["add_all"] else sum(min(c["frontier"], r * c["topk"]) for r in rows)
    return min(c["budget"], 1 + grown)


def work(case):
    esz = 2 if case["dtype"] == "bf16" else 4
    if case["kind"] == "argmax":
        n = case["rows"] * case["vocab"]
        return {"bytes": n * esz + case["rows"] * 4, "flops": n}
    b, nw = case["batch"], _final_nodes(case)
    if case["kind"] == "mask":
        return {"bytes": b * nw * case["kv_len"] * (2 if case["out"] == "bf16" else 4), "flops": b * nw * case["kv_len"]}
    draft = b * sum(_rows_per_level(case)) * case["vocab"] / case["shards"]
    walked = 1 + min(sum(ACCEPT_LEVELS) / 2, case["depth"])
    target = b * (walked if case["kind"] in ("lazy", "host") else nw) * case["vocab"] / case["shards"]
    # per draft element: maximum, exponential, two sums; per target element: maximum
    results = b * nw * (3 * 4 + 8 * ((nw + 63) // 64) + 4 * (case["depth"] + 1))
    records = 288 * b * sum(_rows_per_level(case)) * case["shards"] if case["kind"] == "shard" else 0
    return {"bytes": (draft + target) * esz + results + records, "flops": 6 * draft + target}


def tolerance(case):
    """The sums over a row are 32-bit; a node or token can change places only where two confidences agree that far."""
    if case["kind"] in ("argmax", "mask"):
        return "exact"
    return {"rel": 1e-5, "max": 1e-4, "differ": 5e-3}


# ---------------------------------------------------------------------------- inputs and calls

def _dtype(name):
    return torch.bfloat16 if name == "bf16" else torch.float32


def _room(batch, rows, vocab, dtype):
    """[batch, rows, vocab] whose rows start on 16-byte boundaries, as the library asks."""
    pad = 16 // (2 if dtype == torch.bfloat16 else 4)
    return torch.zeros((batch, rows, -(-vocab // pad) * pad), dtype=dtype, device="cuda")[:, :, :vocab]


def _config(c):
    w1, b1, w2, b2 = c2t_inputs.classifier_weights(c["hidden"], seed=0)
    return c2t.Config(batch=c["batch"], vocab=c["vocab"], dtype=c2t.BF16 if c["dtype"] == "bf16" else c2t.F32,
                      max_depth=c["depth"], topk=c["topk"], frontier_cap=c["frontier"], budget=c["budget"],
                      threshold=c["threshold"], entropy_top_m=c["top_m"],
                      classifier=c2t.CLS_MLP if c["classifier"] == "mlp" else c2t.CLS_IDENTITY_JOINT,
                      hidden=c["hidden"], w1=w1, b1=b1, w2=w2, b2=b2,
                      tree_add=c2t.ADD_ALL_SURVIVORS if c["add_all"] else c2t.ADD_FRONTIER)


def _plant_paths(ctx, target, vocab, seed):
    """Raises one logit per node on a path of every final tree, so that the walk accepts the path."""
    torch.cuda.synchronize()
    ver = {k: ctx.verify[k].cpu().tolist() for k in ("retrieve", "n_leaves", "tokens")}
    where, lo, hi = [], *ACCEPT_LEVELS
    for b in range(ctx.B):
        rows = ver["retrieve"][b][:max(1, ver["n_leaves"][b])]
        deepest = sorted(([x for x in r if x >= 0] for r in rows), key=len)
        chain = deepest[-1 - (seed + b) % min(3, len(deepest))][:1 + lo + (seed + b) % (hi - lo + 1)]
        for here, nxt in zip(chain, chain[1:]):
            where.append((b, here, ver["tokens"][b][nxt]))
    if where:
        i = torch.tensor(where, device=target.device).T
        target[i[0], i[1], i[2]] = 200.0


def prepare(case, seed):
    c, dt, dev = case, _dtype(case["dtype"]), "cuda"
    gen = torch.Generator(device=dev)
    gen.manual_seed(c2t_inputs.key_seed(seed))
    if c["kind"] == "argmax":
        logits = _room(1, c["rows"], c["vocab"], dt)[0]
        logits.copy_(torch.randn(logits.shape, generator=gen, device=dev, dtype=dt) * 3)
        return {"case": c, "logits": logits, "out": torch.zeros(c["rows"], dtype=torch.int32, device=dev)}

    ctx = c2t.Context(_config(c))
    B, F, V, D, Nw = ctx.B, ctx.F, ctx.V, ctx.D, ctx.Nw
    view = ctx.c2t_get_view()
    for name in ("tree_C", "cand_H"):                   # confidences of all nodes, entropies at the last level
        view[name].zero_()                              # (the parts that no step writes)
    draft = []
    for l in range(D):
        t = _room(B, F, V, dt)
        t.copy_(c2t_inputs.draft_logits(B, F, V, 0, l, dt, scale=c["scale"], device=dev, master=seed))
        draft.append(t)
    target = _room(B, Nw, V, dt)
    target.copy_(c2t_inputs.target_logits(B, Nw, V, 0, dt, scale=c["scale"], device=dev, master=seed))
    root = c2t_inputs.root_tokens(B, V, master=seed).to(dev)
    if c["kind"] == "mask":
        prefix = torch.randint(c["prefix"] // 2, c["prefix"] + 1, (B,), generator=gen, device=dev, dtype=torch.int32)
    else:
        prefix = c2t_inputs.prefix_lengths(B, master=seed).to(dev)
    ctx.decode_step(draft, target, root, prefix)
    _plant_paths(ctx, target, V, seed)
    s = {"case": c, "ctx": ctx, "draft": draft, "target": target, "root": root, "prefix": prefix,
         "views": [view["tree_C"], view["cand_H"]]}
    if c["kind"] == "mask":
        return {"case": c, "ctx": ctx, "prefix": prefix, "root": root,      # the step's arrays stay the caller's
                "out": torch.zeros((B, Nw, c["kv_len"]), dtype=_dtype(c["out"]), device=dev)}
    if c["kind"] == "host":
        s.update(draft=[t.contiguous().cpu().pin_memory() for t in draft], target=target.contiguous().cpu().pin_memory(),
                 root=root.cpu().pin_memory(), prefix=prefix.cpu().pin_memory())
        s["stage"], s["results"] = ctx.host_step_buffers()
    if c["kind"] == "shard":
        s.update(_prepare_shard(c, ctx, draft, target, root, prefix))
    return s


def _prepare_shard(c, ctx, draft, target, root, prefix):
    """This rank's token range of every row, and what the all-gathers bring from the other ranks (computed here range
    by range): records [shards, B, F] per level, keys [shards, B, Nw]."""
    ranges = shard_ranges(c["vocab"], c["shards"], 2 if c["dtype"] == "bf16" else 4)
    me = len(ranges) // 2
    records = [ctx.new_row_records(len(ranges)) for _ in range(ctx.D)]
    keys = torch.zeros((len(ranges), ctx.B, ctx.Nw), dtype=torch.int64, device="cuda")
    for r, (v0, v1) in enumerate(ranges):
        for l in range(ctx.D):       # a level's records follow from the level's rows alone; the frontiers from whole rows
            ctx.c2t_begin_step(root, prefix)
            for k in range(l):
                ctx.c2t_expand_prune_level(k, draft[k])
            ctx.c2t_expand_level_shard(l, draft[l][:, :, v0:v1])
            ctx.c2t_export_row_records(l, v0, records[l][r])
    ctx.c2t_begin_step(root, prefix)
    for l in range(ctx.D):
        ctx.c2t_expand_prune_level(l, draft[l])
    ctx.c2t_prune(c2t.FINAL)
    ctx.c2t_build_verify()
    for r, (v0, v1) in enumerate(ranges):
        ctx.c2t_argmax_shard(target[:, :, v0:v1], v0, keys[r])
    v0, v1 = ranges[me]
    mine = []
    for t in draft + [target]:
        part = _room(t.shape[0], t.shape[1], v1 - v0, t.dtype)
        part.copy_(t[:, :, v0:v1])
        mine.append(part)
    return {"draft": mine[:-1], "target": mine[-1], "records": records, "keys": keys, "me": me, "begin": v0}


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "argmax":
        c2t.c2t_row_argmax_static(s["logits"], s["out"])
        return s["out"]
    ctx = s["ctx"]
    if kind == "mask":
        ctx.c2t_dense_mask(s["out"])
        return s["out"]
    if kind == "host":
        ctx.c2t_decode_step_host(s["draft"], s["target"], s["root"], s["prefix"], s["results"], s["stage"])
        return [s["results"], s["views"]]
    if kind == "step":
        ctx.decode_step(s["draft"], s["target"], s["root"], s["prefix"])
    elif kind == "lazy":
        ctx.c2t_begin_step(s["root"], s["prefix"])
        for l in range(ctx.D):
            ctx.c2t_expand_prune_level(l, s["draft"][l])
        ctx.c2t_prune(c2t.FINAL)
        ctx.c2t_build_verify()
        ctx.c2t_accept_lazy(s["target"])
    else:
        ctx.c2t_begin_step(s["root"], s["prefix"])
        for l in range(ctx.D):
            ctx.c2t_expand_level_shard(l, s["draft"][l])
            ctx.c2t_export_row_records(l, s["begin"], s["records"][l][s["me"]])
            ctx.c2t_prune_gathered(l, s["records"][l])
        ctx.c2t_prune(c2t.FINAL)
        ctx.c2t_build_verify()
        ctx.c2t_argmax_shard(s["target"], s["begin"], s["keys"][s["me"]])
        ctx.c2t_accept_gathered(s["keys"])
    return [ctx.verify, ctx.accepted, ctx.frontier["count"], s["views"]]
