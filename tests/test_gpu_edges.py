"""GPU parity at the edges of the kernels' tiles and dispatch rules: chunks of the expand pass, rows in registers and rows that are streamed, the K for which it takes its
bound from half columns, its selection in order, the sizes of the lazy walk's clusters, the rerank of large trees, the short
and long rows of the arg-max pass, the mask's 16-byte vectors, the host step."""
import numpy as np
import pytest
import torch

import c2t_inputs
import oracle
import paper_2502_13652_b200 as c2t
from parity_util import gen_inputs, make_configs, run_and_compare, special_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2502_13652_b200 import build
    build.build()
    oracle.build()


def step(B, V, D, K, F, N, beta, dtype, draft=None, **kw):
    ocfg, gcfg = make_configs(B, V, D, K, F, N, beta, dtype, **kw)
    dr, target, root, prefix = gen_inputs(B, V, D, F, c2t.c2t_final_width(gcfg), dtype)
    pad = -(-V // 8) * 8

    def rows(t):                                       # rows on 16-byte boundaries
        buf = torch.zeros(t.shape[0], t.shape[1], pad, dtype=dtype, device="cuda")
        buf[:, :, :V] = t.cuda()
        return buf[:, :, :V]

    dr = draft if draft is not None else dr
    rep = run_and_compare(ocfg, gcfg, dr, target, root, prefix, draft_dev=[rows(t) for t in dr], target_dev=rows(target))
    assert rep.status_bits == 0


# a chunk is 256 vectors: 2048 bf16 or 1024 fp32 tokens; two chunks share a word of cells; 12 warps stream
@pytest.mark.parametrize("dtype,chunk", [(torch.bfloat16, 2048), (torch.float32, 1024)])
@pytest.mark.parametrize("V", ["7", "1-1", "1", "1+1", "2+5", "3", "12+1", "64", "65-3"])
def test_vocabulary_around_chunk_edges(dtype, chunk, V):
    n, plus = (V + "+0").split("+")[:2] if "+" in V else ((V.split("-")[0], "-" + V.split("-")[1]) if "-" in V else (V, "0"))
    v = 7 if V == "7" else int(n) * chunk + int(plus)
    step(3, v, 3, 4, 5, 14, 0.0, dtype, classifier="identity")


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("K", [16, 17, 32])
def test_widths_of_the_selection(dtype, K):
    step(2, 9000, 2, K, 3, 20, 0.0, dtype, classifier="identity")


@pytest.mark.parametrize("B,K,F", [(1, 7, 7), (15, 10, 10)])
def test_few_frontier_nodes_with_long_rows(B, K, F):
    """A row lies in many chunks; its cells and records must stay clear of each other and of the arg-max keys behind them, which the
    acceptance calls (compared here too) take their maxima from."""
    step(B, 128256, 3, K, F, 40, 0.5, torch.float32)


@pytest.mark.parametrize("dtype,V,M", [(torch.bfloat16, 8192, 1000), (torch.float32, 4099, 700), (torch.bfloat16, 32768, 4000),
                                       (torch.float32, 32768, 7000), (torch.bfloat16, 32776, 5000), (torch.bfloat16, 1003, 1002)])
def test_truncated_entropy_of_rows_read_again(dtype, V, M):
    """M so large that nothing is set aside: rows that fit in shared memory as a whole, up to the last that does, and the next."""
    step(3, V, 3, 4, 3, 10, 0.0, dtype, M=M)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_rows_with_more_candidates_than_the_pool(dtype):
    """Well over a hundred equal largest values in scattered cells: more than the pool of a row holds, so the row is taken in
    token order.  Such a row's candidates have the probability 1 / count, and with equal counts in two rows children of
    different rows would tie to 1e-6, where either order is right; the counts here differ by 4 % or more from row to row."""
    B, V, F, D = 2, 24000, 4, 2
    g = torch.Generator().manual_seed(3)
    draft = []
    for _ in range(D):
        x = torch.randn(B, F, V, generator=g)
        for b in range(B):
            for j in range(F):
                x[b, j, ::80 + 9 * (F * b + j)] = 20.0
        draft.append(x.to(dtype))
    step(B, V, D, 6, F, 12, 0.0, dtype, draft=draft, classifier="identity")


@pytest.mark.parametrize("dtype,V", [(torch.bfloat16, 8200), (torch.float32, 4100), (torch.bfloat16, 40003), (torch.float32, 16389)])
@pytest.mark.parametrize("B", [1, 37, 75, 149])
def test_lazy_walk_equals_the_walk_over_all_rows(B, V, dtype):
    """Clusters of 8, 8 or 4, 2 and 1 CTAs per sequence on a chip of 148 SMs; short and long, whole and ragged rows."""
    D, K, F, N = 3, 4, 3, 9
    _, gcfg = make_configs(B, V, D, K, F, N, 0.0, dtype, classifier="identity")
    ctx = c2t.Context(gcfg)
    pad = -(-V // 8) * 8
    g = torch.Generator(device="cuda").manual_seed(B)
    draft = [torch.randn(B, F, pad, device="cuda", generator=g).to(dtype)[:, :, :V] for _ in range(D)]
    target = torch.randn(B, ctx.Nw, pad, device="cuda", generator=g).to(dtype)[:, :, :V]
    zeros = torch.zeros(B, dtype=torch.int32, device="cuda")
    ctx.decode_step(draft, target, zeros, zeros)
    ver = {k: v.cpu() for k, v in ctx.verify.items()}
    for b in range(B):                                  # a path of every length, the last token near the row's end
        row = [int(x) for x in ver["retrieve"][b, b % int(ver["n_leaves"][b])] if x >= 0][:1 + b % (D + 1)]
        for here, nxt in zip(row, row[1:]):
            target[b, here, int(ver["tokens"][b, nxt])] = 50.0
        target[b, row[-1], V - 1] = 60.0
    ctx.c2t_accept(target)
    torch.cuda.synchronize()
    want = {k: v.clone() for k, v in ctx.accepted.items()}
    amax = ctx.c2t_get_view()["node_argmax"].clone()
    assert torch.equal(amax.cpu(), target.float().cpu().max(dim=2).indices.to(torch.int32)[:, :ctx.Nw].where(
        torch.arange(ctx.Nw)[None, :] < ver["n_nodes"][:, None], torch.tensor(-1, dtype=torch.int32)))
    assert int(want["accept_len"].max()) >= min(B - 1, D - 1)
    ctx.c2t_accept_lazy(target)
    torch.cuda.synchronize()
    for k, v in want.items():
        assert torch.equal(ctx.accepted[k], v), k
    on_path = torch.zeros_like(amax, dtype=torch.bool)
    path = want["path"].long()
    on_path.scatter_(1, path.clamp(min=0), True)
    assert torch.equal(ctx.c2t_get_view()["node_argmax"], torch.where(on_path, amax, -1))
    ctx.close()


@pytest.mark.parametrize("N,wstd", [(20, 0.1), (400, 0.1), (20, 0.0), (1, 0.1)])
def test_rerank_of_a_large_tree(N, wstd):
    """511 nodes (more than a warp ranks one by one), with distinct confidences and with all of them equal."""
    step(2, 3000, 6, 10, 10, N, 0.0, torch.float32, tree_add="all", wstd=wstd)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("kv", [1, 7, 40, 133, 256])
def test_mask_vectors(dtype, kv):
    """Rows that start on every alignment, end inside the prefix, inside the tree and behind it."""
    B, V, D, K, F, N = 3, 2000, 4, 4, 4, 13
    _, gcfg = make_configs(B, V, D, K, F, N, 0.0, torch.bfloat16, classifier="identity")
    ctx = c2t.Context(gcfg)
    draft = [torch.randn(B, F, V, device="cuda").to(torch.bfloat16) for _ in range(D)]
    prefix = torch.tensor([0, 33, 128], dtype=torch.int32)
    ctx.c2t_begin_step(torch.zeros(B, dtype=torch.int32, device="cuda"), prefix.cuda())
    for l in range(D):
        ctx.c2t_expand_level(l, draft[l]); ctx.c2t_prune(l)
    ctx.c2t_prune(c2t.FINAL); ctx.c2t_build_verify()
    out = torch.full((B, ctx.Nw, kv), 7.0, dtype=dtype, device="cuda")
    ctx.c2t_dense_mask(out)
    bits = ctx.verify["mask_bits"].cpu().numpy()
    got = out.float().cpu().numpy()
    for b in range(B):
        for i in range(ctx.Nw):
            on = [c < prefix[b] or (c - prefix[b] < 64 and int(bits[b, i, 0]) >> int(c - prefix[b]) & 1) for c in range(kv)]
            assert np.array_equal(got[b, i], np.where(np.array(on, dtype=bool), 0.0, -np.inf)), (b, i)
    ctx.close()


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("N", [16, 3])
def test_host_step_ways(pinned, N):
    """Pinned or pageable host buffers; two staging buffers for the levels, or one (N < F)."""
    B, V, D, K, F = 3, 4096, 4, 5, 4
    _, gcfg = make_configs(B, V, D, K, F, N, 0.3, torch.bfloat16)
    draft, target, root, prefix = gen_inputs(B, V, D, F, c2t.c2t_final_width(gcfg), torch.bfloat16)
    ctx = c2t.Context(gcfg)
    ctx.decode_step([t.cuda() for t in draft], target.cuda(), root.cuda(), prefix.cuda())
    torch.cuda.synchronize()
    want = {k: v.cpu().clone() for k, v in list(ctx.verify.items())[:2] + list(ctx.accepted.items())}
    stage, results = ctx.host_step_buffers()
    pin = (lambda t: t.pin_memory()) if pinned else (lambda t: t.contiguous())
    for _ in range(2):
        ctx.c2t_decode_step_host([pin(t) for t in draft], pin(target), root, prefix, results, stage)
        for k, w in want.items():
            assert torch.equal(results[k], w), k
    ctx.close()


def far_rows(kind, B, F, V, dtype, seed):
    """Rows whose warps first meet values far below the rest: a head of -80, then a body near -11, then one peak; or a body 60 to
    69 above the head and a peak of 1e9."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    noise = torch.rand(B, F, V, device="cuda", generator=g)
    if kind == "masked_head":
        x = -11.2 + 0.1 * noise
        x[:, :, :2 * V // 5] = -80.0
        x[:, :, V - 3000:] = -90.0
        x[:, :, V - 1500] = 8.5
    else:
        x = 60.0 + 9.0 * noise
        x[:, :, :2 * V // 5] = noise[:, :, :2 * V // 5]
        x[:, :, V - 1500] = 1e9
    return x.to(dtype)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("kind", ["masked_head", "jump"])
def test_rows_with_a_head_far_below_the_rest(dtype, kind):
    """Enough chunks per row and rows per CTA that a warp meets all three parts; the sums of the body must survive the peak."""
    B, V = 160, 65536 if dtype == torch.float32 else 131072
    ocfg, gcfg = make_configs(B, V, 1, 10, 1, 0, 0.0, dtype, classifier="identity")
    _, target, root, prefix = gen_inputs(1, V, 1, 1, c2t.c2t_final_width(gcfg), dtype)
    rep = run_and_compare(ocfg, gcfg, None, None, root.expand(B).contiguous(), prefix.expand(B).contiguous(), seqs=[0, 9, 77, 159],
                          draft_dev=[far_rows(kind, B, 1, V, dtype, 3)], target_dev=target.cuda().expand(B, -1, -1).contiguous())
    assert rep.status_bits == 0


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("scale", [4.0, 8.0])
def test_error_of_probabilities_and_entropies(dtype, scale):
    """One level of whole rows.  A weight 2^t carries the error of `ex2.approx` (2^-22 at most) and the rounding of t (2^-25 for the
    t in [-1, 0] of the largest ones), fp32 additions 2^-24 a few times over: 4e-7 in a probability.  An entropy is ln(1 + S) plus a sum
    of weights times their logarithm, each with that error: 1e-6."""
    B, V = 16, 128256
    ocfg, gcfg = make_configs(B, V, 1, 10, 10, 12, 0.0, dtype)
    draft, target, root, prefix = gen_inputs(B, V, 1, 10, c2t.c2t_final_width(gcfg), dtype, scale=scale, device="cuda")
    rep = run_and_compare(ocfg, gcfg, None, None, root, prefix, draft_dev=draft, target_dev=target)
    assert rep.status_bits == 0 and rep.max_rel_p < 4e-7 and rep.max_rel_H < 1e-6


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_static_argmax_of_cut_rows_and_after_an_overlap(dtype):
    """Rows cut between thread blocks in every way: one row over many of them, rows that begin or end with a span, whole rows between
    two cut ones, rows shorter than a span.  Then calls on two streams that may overlap: what they return is undefined, what
    later calls return is not."""
    vec = 8 if dtype == torch.bfloat16 else 4
    g = torch.Generator(device="cuda").manual_seed(2)
    shapes = [(1, 262144), (1, 5), (3, 1024 * vec), (7, 1536 * vec), (40, 128256), (297, 1023 * vec + 3), (4096, 1000)]

    def check():
        for rows, V in shapes:
            x = torch.randn(rows, -(-V // 8) * 8, device="cuda", generator=g).to(dtype)[:, :V]
            at = torch.randint(0, V, (rows,), device="cuda", generator=g)
            x[torch.arange(rows, device="cuda"), at] = 9.0
            out = torch.full((rows,), -7, dtype=torch.int32, device="cuda")
            c2t.c2t_row_argmax_static(x, out)
            assert torch.equal(out, at.to(torch.int32)), (rows, V)

    check()
    x = torch.randn(64, 128256, device="cuda", generator=g).to(dtype)
    outs = [torch.zeros(64, dtype=torch.int32, device="cuda") for _ in range(2)]
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(50):
        for s, o in zip(streams, outs):
            c2t.c2t_row_argmax_static(x, o, s)
    torch.cuda.synchronize()
    check()


@pytest.mark.parametrize("classifier", ["mlp", "identity"])
def test_first_step_on_a_stream_of_its_own(classifier):
    """The default stream is busy when the context is made; the first step runs on a stream that does not wait for it."""
    B, V, D, K, F, N = 2, 32000, 3, 5, 4, 12
    _, gcfg = make_configs(B, V, D, K, F, N, 0.0, torch.float32, classifier=classifier)
    draft, target, root, prefix = gen_inputs(B, V, D, F, c2t.c2t_final_width(gcfg), torch.float32)
    draft = [t.cuda() for t in draft]; target = target.cuda(); root = root.cuda(); prefix = prefix.cuda()
    side = torch.cuda.Stream()
    outs = []
    for busy in (False, True):
        torch.full((64 << 20,), -1, dtype=torch.int32, device="cuda")              # (the next workspace is not all zeros)
        torch.cuda.synchronize()
        if busy:
            torch.cuda._sleep(100_000_000)
        ctx = c2t.Context(gcfg)
        with torch.cuda.stream(side):
            ctx.decode_step(draft, target, root, prefix)
        torch.cuda.synchronize()
        assert ctx.c2t_status()[0] == 0
        outs.append([v.clone() for v in list(ctx.verify.values()) + list(ctx.accepted.values())])
        ctx.close()
    for a, b in zip(*outs):
        assert torch.equal(a, b)


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("B,M,N", [(1, 0, 16), (2, 0, 3), (3, 64, 16), (5, 0, 16)])
def test_host_step_leaves_what_the_calls_leave(B, M, N, pinned):
    """One and two sequences, the truncated entropy, a budget below the frontier: results, the arg-max of every final node and the
    staged rows are those of the calls one by one, whatever memory the rows come from."""
    V, D, K, F = 8192, 4, 5, 4
    _, gcfg = make_configs(B, V, D, K, F, N, 0.3, torch.bfloat16, M=M)
    draft, target, root, prefix = gen_inputs(B, V, D, F, c2t.c2t_final_width(gcfg), torch.bfloat16)
    ctx = c2t.Context(gcfg)
    view = ctx.c2t_get_view()
    ctx.decode_step([t.cuda() for t in draft], target.cuda(), root.cuda(), prefix.cuda())
    want = {k: v.cpu().clone() for k, v in list(ctx.verify.items())[:2] + list(ctx.accepted.items())}
    amax = view["node_argmax"].clone()
    assert int((amax >= 0).sum()) == int(want["n_nodes"].sum())
    stage, results = ctx.host_step_buffers()
    pin = (lambda t: t.pin_memory()) if pinned else (lambda t: t.contiguous())
    for _ in range(2):
        view["node_argmax"].fill_(-7)
        torch.cuda.synchronize()
        ctx.c2t_decode_step_host([pin(t) for t in draft], pin(target), root, prefix, results, stage)
        for k, w in want.items():
            assert torch.equal(results[k], w), k
        assert torch.equal(view["node_argmax"], amax)
        assert torch.equal(stage["target"].cpu(), target) and torch.equal(stage["draft"].cpu(), draft[D - 1])
    ctx.close()


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("mask", [float("-inf"), torch.finfo(torch.float32).min, -1e9, -10000.0, 0.0, 7.0])
@pytest.mark.parametrize("V", [4096, 30000, 33 * 1024 + 5])
def test_rows_of_one_value_but_for_a_few(dtype, mask, V):
    """The K-th largest is the value that fills the row: the lowest tokens that hold it, and before them what lies above it, also by
    less than a bf16 step (an fp32 cell is rounded to one) and in the row's last chunk."""
    B, K = 6, 10
    x = torch.full((B, 1, V), mask)
    g = torch.Generator().manual_seed(1)
    for b in range(B):
        at = torch.randperm(V, generator=g)[:b + 3]
        x[b, 0, at] = 20.0 + torch.arange(b + 3)
        if mask > -1e30 and dtype == torch.float32:     # just above, early and late
            x[b, 0, V - 1 - 700 * b] = torch.nextafter(torch.tensor(mask), torch.tensor(100.0)) + abs(mask) * 1e-6
            x[b, 0, 2 * b] = torch.nextafter(torch.tensor(mask), torch.tensor(100.0))
    ocfg, gcfg = make_configs(B, V, 1, K, 1, 0, 0.0, dtype, classifier="identity")
    _, target, root, prefix = gen_inputs(B, V, 1, 1, c2t.c2t_final_width(gcfg), dtype)
    pad = -(-V // 8) * 8

    def rows(t):
        buf = torch.zeros(B, t.shape[1], pad, dtype=dtype, device="cuda")
        buf[:, :, :V] = t.cuda()
        return buf[:, :, :V]

    x = x.to(dtype)
    rep = run_and_compare(ocfg, gcfg, [x], target, root, prefix, draft_dev=[rows(x)], target_dev=rows(target))
    assert rep.status_bits == 0


# Rows in registers: a block of 256 threads holds 2048 vectors of 16 bytes, eight of them 16384; beyond that blocks of 512, up to 32768;
# longer rows are streamed.
@pytest.mark.parametrize("dtype,V", [(torch.bfloat16, 16384), (torch.bfloat16, 16385), (torch.bfloat16, 131072), (torch.bfloat16, 131073),
                                     (torch.float32, 8191), (torch.float32, 8193), (torch.float32, 65537), (torch.float32, 131072),
                                     (torch.float32, 131073)])
def test_rows_around_a_block_of_registers(dtype, V):
    step(1, V, 2, 3, 3, 6, 0.0, dtype, classifier="identity")


@pytest.mark.parametrize("dtype,chunk", [(torch.bfloat16, 2048), (torch.float32, 1024)])
@pytest.mark.parametrize("n,plus", [(1, -1), (1, 1), (2, 5), (12, 1)])
def test_streamed_rows_around_chunk_edges(dtype, chunk, n, plus):
    """Level 1 has 320 rows, too many for the registers (296 blocks): cut into chunks and streamed."""
    step(160, n * chunk + plus, 2, 2, 2, 4, 0.0, dtype, classifier="identity")


@pytest.mark.parametrize("dtype,V", [(torch.bfloat16, 4099), (torch.float32, 2050), (torch.bfloat16, 30000)])
def test_equal_largest_values_around_what_a_block_lists(dtype, V):
    """40 to 146 equal largest values in a row: a row of one block lists 128 keys, the blocks of a cluster 64 each and 128 together."""
    B, K = 75, 6
    g = torch.Generator().manual_seed(7)
    x = torch.randn(B, 1, V, generator=g)
    for b in range(B):
        n = 40 + b + (32 if b >= 40 else 0)
        at = torch.randperm(V // 4 if b % 3 == 0 else V, generator=g)[:n]
        x[b, 0, at] = 20.0
    step(B, V, 1, K, 1, 0, 0.0, dtype, draft=[x.to(dtype)], classifier="identity")


@pytest.mark.parametrize("B", [2, 60])
def test_cap_between_confidences_with_equal_upper_halves(B):
    """Sixteen children whose fp32 logits of 0.5 to 1 are one unit in the last place apart (6e-8 in their probabilities): the upper 32 bits of
    neighbouring confidences, 20 of the mantissa, are equal, so the lower ones decide the frontier cap in their middle."""
    V, F, D = 9000, 8, 2
    g = torch.Generator().manual_seed(5)
    draft = []
    for _ in range(D):
        x = torch.randn(B, F, V, generator=g) - 6.0
        for b in range(B):
            for j in range(F):
                at = torch.randperm(V, generator=g)[:16]
                x[b, j, at] = 0.5 + 0.06 * j + torch.arange(16) * 2.0 ** -24
        draft.append(x)
    step(B, V, D, 16, F, 12, 0.0, torch.float32, draft=draft, classifier="identity")


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("B,V,K,F", [(2, 23862, 14, 10), (60, 23862, 14, 10), (2, 9000, 32, 32), (30, 9000, 32, 32), (20, 9000, 12, 10),
                                     (2, 128256, 16, 20)])
def test_cap_takes_the_first_by_confidence_and_index(B, V, K, F, sign):
    """Several levels with K above F or near it: joint probabilities shrink from level to level, and a row's children have confidences that
    share up to all of their upper bits.  What is selected must be the F first under (C desc, index asc), by the confidences that the
    kernels themselves wrote; with sign -1 the larger ones have the larger index.  The two launches at a level and the one that does both."""
    D = 4
    w1, b1, w2, b2 = c2t_inputs.classifier_weights(16, seed=0)
    _, cfg = make_configs(B, V, D, K, F, 40, 0.0, torch.float32, weights=(w1, b1, sign * w2, b2))
    draft, _, root, prefix = gen_inputs(B, V, D, F, 8, torch.float32, device="cuda")
    pad = -(-V // 4) * 4
    draft = [torch.nn.functional.pad(t.cuda(), (0, pad - V))[:, :, :V] for t in draft]
    ctx = c2t.Context(cfg)
    undecided = turned = 0
    for two in (False, True):
        ctx.c2t_begin_step(root.cuda(), prefix.cuda())
        for l in range(D):
            if two:
                ctx.c2t_expand_level(l, draft[l]); ctx.c2t_prune(l)
            else:
                ctx.c2t_expand_prune_level(l, draft[l])
            view = ctx.c2t_get_view()
            n, flags, C = (view[k].cpu().numpy() for k in ("cand_n", "cand_flags", "cand_C"))
            for b in range(B):
                m = n[b]
                keep, c = (flags[b, :m] & 1) != 0, C[b, :m]
                assert m > 0 and keep.all()
                order = np.lexsort((np.arange(m), -c))
                want = np.zeros(m, dtype=bool)
                want[order[:F]] = True
                assert np.array_equal(want, (flags[b, :m] & 2) != 0), (l, b)
                if m > F:
                    upper = c.view(np.uint64) >> np.uint64(32)
                    undecided += upper[order[F - 1]] == upper[order[F]]
                    by_upper = np.lexsort((np.arange(m), -upper.astype(np.int64)))
                    turned += set(by_upper[:F]) != set(order[:F])
    ctx.close()
    if K > F:
        assert undecided > B and (turned > 0 or sign > 0), (undecided, turned)


@pytest.mark.parametrize("B,V,dtype", [(1, 32000, torch.float32), (5, 9001, torch.bfloat16), (40, 20000, torch.bfloat16)])
def test_step_in_one_call_equals_single_calls(B, V, dtype):
    """c2t_decode_step (levels in one launch, or streamed and pruned) against separate expand and prune calls: bit for bit."""
    D, K, F, N = 4, 6, 9, 30
    _, cfg = make_configs(B, V, D, K, F, N, 0.3, dtype)
    pad = -(-V // 8) * 8
    draft, target, root, prefix = gen_inputs(B, V, D, F, c2t.c2t_final_width(cfg), dtype)

    def rows(t):
        buf = torch.zeros(t.shape[0], t.shape[1], pad, dtype=dtype, device="cuda")
        buf[:, :, :V] = t.cuda()
        return buf[:, :, :V]

    draft = [rows(t) for t in draft]; target = rows(target); root = root.cuda(); prefix = prefix.cuda()
    ctx = c2t.Context(cfg)
    got = []
    for single in (False, True, None):
        if single is None:
            ctx.c2t_decode_step(draft, target, root, prefix)
        elif single:
            ctx.c2t_begin_step(root, prefix)
            for l in range(D):
                ctx.c2t_expand_level(l, draft[l]); ctx.c2t_prune(l)
            ctx.c2t_prune(c2t.FINAL); ctx.c2t_build_verify(); ctx.c2t_accept(target)
        else:
            ctx.decode_step(draft, target, root, prefix)
        torch.cuda.synchronize()
        v = ctx.c2t_get_view()
        live = torch.arange(ctx.cap, device="cuda")[None, :] < v["tree_n"][:, None]
        got.append([t.clone() for t in list(ctx.verify.values()) + list(ctx.accepted.values()) + list(ctx.frontier.values())] +
                   [v["tree_n"].clone(), torch.where(live, v["tree_logP"], 0.0), torch.where(live, v["tree_C"], 0.0)])
    assert ctx.c2t_status()[0] == 0 and int(got[0][-3].max()) > 1
    for a, b, c in zip(*got):
        assert torch.equal(a, b) and torch.equal(a, c)
    ctx.close()


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_equal_values_in_the_lane_of_the_maximum(dtype):
    """A row in registers whose finite values all belong to one thread (vectors 256 apart): the maximum, which it sums again without, and
    n equal others.  A weight may be off by what `ex2.approx` is, but n equal weights are n times one of them: the lane's elements are
    added in fp32 two at a time, which is exact here, and else in fp64."""
    V = 131072 if dtype == torch.bfloat16 else 65536   # eight blocks of 256 threads with 8 vectors each
    vec = 8 if dtype == torch.bfloat16 else 4
    _, cfg = make_configs(1, V, 1, 4, 1, 0, 0.0, dtype, classifier="identity")
    ctx = c2t.Context(cfg)
    record = ctx.new_row_records()[0]
    zero = torch.zeros(1, dtype=torch.int32, device="cuda")
    at = torch.tensor([2048 * 2 + 256 * k + 7 for k in range(8)])[:, None] * vec + torch.arange(vec)
    at = at.flatten().cuda()
    S = {}
    for n in [1, 3, 7, 13, 21, 31] + [47, 63] * (vec == 8):
        x = torch.full((1, 1, V), float("-inf"), dtype=dtype, device="cuda")
        x[0, 0, at[1:1 + n]] = 1.6875
        x[0, 0, at[0]] = 3.0
        ctx.c2t_begin_step(zero, zero)
        ctx.c2t_expand_level_shard(0, x)
        ctx.c2t_export_row_records(0, 0, record)
        S[n] = float(record[0, 0, 8:16].cpu().view(torch.float64))
    ctx.close()
    assert abs(S[1] / np.exp(-1.3125) - 1) < 5e-7
    for n in S:
        assert abs(S[n] / (n * S[1]) - 1) < 1e-13, (n, S[n] / (n * S[1]) - 1)


def blocks_of_a_row(V, dtype, rows, K):
    """How the level's rows are cut: blocks per row in registers, or 0 where they are streamed."""
    import ctypes
    from paper_2502_13652_b200 import build
    plan = ctypes.CDLL(build.build(debug_bounds=True)).c2t_debug_row_cluster
    plan.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    return plan(V, 2 if dtype == torch.bfloat16 else 4, rows, K, torch.cuda.get_device_properties(0).multi_processor_count)


def streamed_row(kind, V, b, dtype):
    g = torch.Generator().manual_seed(b)
    if isinstance(kind, float):                        # one value but for a few, just above it too
        x = torch.full((V,), kind)
        at = torch.randperm(V, generator=g)[:b % 6 + 3]
        x[at] = 20.0 + torch.arange(b % 6 + 3)
        if kind > -1e30 and dtype == torch.float32:
            up = torch.nextafter(torch.tensor(kind), torch.tensor(100.0))
            x[V - 1 - 70 * (b % 6)] = up + abs(kind) * 1e-6
            x[2 * (b % 6)] = up
    elif kind == "equal":                              # more equal largest values than the pool of a row holds
        x = torch.randn(V, generator=g)
        x[::max(1, V // (150 + 9 * (b % 6)))] = 20.0
    else:
        x = special_rows(kind, 1, 1, V, torch.float32)[0, 0] + 0.25 * (b % 6)
    return x.to(dtype)


# many rows in two launches (fp32: the long ones' cells in shared memory, at 96 chunks of 1024 tokens and below), few long ones, two sequences
# in one launch
@pytest.mark.parametrize("dtype,B,V", [(torch.bfloat16, 320, 4096), (torch.bfloat16, 300, 20003), (torch.bfloat16, 3, 270000), (torch.bfloat16, 2, 270000),
                                       (torch.float32, 320, 4096), (torch.float32, 300, 97280), (torch.float32, 300, 97281), (torch.float32, 3, 140000), (torch.float32, 2, 140000)])
@pytest.mark.parametrize("kind,K", [(float("-inf"), 10), (-1e9, 10), (0.0, 17), (7.0, 32), ("equal", 6), ("two_valued", 32), ("heavy_ties", 10),
                                    ("rising", 17), ("late_jump", 16), ("neg_inf", 32)])
def test_streamed_rows_of_every_kind(dtype, B, V, kind, K):
    assert blocks_of_a_row(V, dtype, B, K) == 0
    ocfg, gcfg = make_configs(B, V, 1, K, 1, 0, 0.0, dtype, classifier="identity")
    pad = -(-V // 8) * 8
    some = torch.zeros(6, 1, pad, dtype=dtype)
    for b in range(6):
        some[b, 0, :V] = streamed_row(kind, V, b, dtype)
    draft = some[torch.arange(B) % 6].cuda()[:, :, :V]
    target = torch.zeros(B, c2t.c2t_final_width(gcfg), 8, dtype=dtype, device="cuda").repeat(1, 1, pad // 8)[:, :, :V]
    ints = torch.zeros(B, dtype=torch.int32)
    seqs = sorted({0, 1, 2, B // 2, B - 3, B - 2, B - 1} & set(range(B)))
    rep = run_and_compare(ocfg, gcfg, None, None, ints, ints, seqs=seqs, draft_dev=[draft], target_dev=target, fused=B <= 2)
    assert rep.status_bits == 0


@pytest.mark.parametrize("dtype,B,V", [(torch.bfloat16, 320, 4096), (torch.float32, 320, 4096), (torch.float32, 4, 140000)])
def test_faults_in_streamed_rows(dtype, B, V):
    assert blocks_of_a_row(V, dtype, B, 4) == 0
    _, cfg = make_configs(B, V, 1, 4, 1, 0, 0.0, dtype, classifier="identity")
    x = torch.randn(B, 1, V, device="cuda").to(dtype)
    x[1, 0, V - 5] = float("nan"); x[2, 0, 17] = float("inf"); x[3, 0] = float("-inf")
    ctx = c2t.Context(cfg)
    ints = torch.zeros(B, dtype=torch.int32, device="cuda")
    ctx.c2t_begin_step(ints, ints)
    ctx.c2t_expand_level(0, x); ctx.c2t_prune(0)
    status = ctx.c2t_status()[1]
    assert status[:4] == [0, c2t.ST_NAN_LOGIT, c2t.ST_POSINF_LOGIT, c2t.ST_ALL_NEGINF] and not any(status[4:])
    assert ctx.frontier["count"].tolist() == [1, 0, 0, 0] + [1] * (B - 4)
    ctx.close()


@pytest.mark.parametrize("K,F", [(10, 20), (20, 20), (32, 24)])
def test_two_sequences_with_streamed_levels_in_one_launch(K, F):
    """The first level in registers, then more long rows than fit there."""
    V, dtype = 128256, torch.bfloat16
    assert blocks_of_a_row(V, dtype, 2, K) > 0 and blocks_of_a_row(V, dtype, 2 * F, K) == 0
    ocfg, gcfg = make_configs(2, V, 4, K, F, 40, 0.5, dtype)
    draft, target, root, prefix = gen_inputs(2, V, 4, F, c2t.c2t_final_width(gcfg), dtype)
    rep = run_and_compare(ocfg, gcfg, draft, target, root, prefix, fused=True)
    assert rep.status_bits == 0
