"""The library built with -DC2T_DEBUG_BOUNDS (every kernel checks the indices of its own writes to queues, pools
and workspace records and reports a failed check as C2T_ST_INTERNAL) must pass the same parity cases without ever
setting that bit.  This is the stand-in for a memory checker.  The variant is a second shared library, selected by
the C2T_LIBRARY environment variable, so the cases run in a child process."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys, torch
sys.path.insert(0, {root!r}); sys.path.insert(0, {tests!r})
import oracle, paper_2502_13652_b200 as c2t
from parity_util import gen_inputs, make_configs, run_and_compare, special_rows
assert c2t.LIB_PATH.endswith("libc2t_debug.so")
oracle.build()
cases = [(2, 32000, 5, 10, 10, 40, 0.5, torch.bfloat16, {{}}),
         (3, 5004, 4, 6, 5, 18, 0.5, torch.float32, {{}}),
         (1, 16384, 3, 32, 32, 100, 0.5, torch.bfloat16, dict(hidden=64, wseed=4)),
         (1, 128256, 4, 8, 16, 40, 0.3, torch.bfloat16, {{}}),
         (2, 4096, 5, 4, 4, 7, 0.0, torch.float32, dict(classifier="identity", tree_add="all")),
         # rows in registers: parts of a vector, one vector more than a block, than eight, than blocks of 256 threads hold
         (2, 1, 2, 1, 1, 3, 0.0, torch.float32, {{}}), (3, 40, 2, 3, 3, 6, 0.0, torch.bfloat16, dict(classifier="identity")),
         (1, 8193, 3, 5, 6, 12, 0.0, torch.float32, dict(classifier="identity")), (1, 65537, 3, 5, 6, 12, 0.0, torch.float32, dict(classifier="identity")),
         (90, 16385, 1, 4, 1, 0, 0.0, torch.bfloat16, dict(classifier="identity")),
         # streamed: in one launch, in two, rows shared by several CTAs and rows inside one, fp32 cells in either place
         (2, 128256, 3, 20, 20, 40, 0.5, torch.bfloat16, {{}}), (3, 140001, 2, 6, 2, 9, 0.0, torch.float32, dict(classifier="identity")),
         (160, 2053, 2, 2, 2, 4, 0.0, torch.bfloat16, dict(classifier="identity")), (150, 97281, 2, 2, 2, 4, 0.0, torch.float32, dict(classifier="identity"))]
for B, V, D, K, F, N, beta, dtype, kw in cases:
    ocfg, gcfg = make_configs(B, V, D, K, F, N, beta, dtype, **kw)
    Nw = c2t.c2t_final_width(gcfg)
    draft, target, root, prefix = gen_inputs(B, V, D, F, Nw, dtype)
    pad = -(-V // 8) * 8
    rows = lambda t: torch.nn.functional.pad(t.cuda(), (0, pad - V))[:, :, :V]
    for fused in (False, True):
        rep = run_and_compare(ocfg, gcfg, draft, target, root, prefix, draft_dev=[rows(t) for t in draft], target_dev=rows(target), fused=fused)
        assert rep.status_bits == 0, rep.status_bits
for kind in ("rising", "uniform", "neg_inf"):
    B, V, D, K, F, N = 2, 20000, 3, 5, 4, 12
    ocfg, gcfg = make_configs(B, V, D, K, F, N, 0.0, torch.bfloat16, classifier="identity")
    Nw = c2t.c2t_final_width(gcfg)
    draft = [special_rows(kind, B, F, V, torch.bfloat16) for _ in range(D)]
    target = special_rows(kind, B, Nw, V, torch.bfloat16)
    root = torch.zeros(B, dtype=torch.int32); prefix = torch.full((B,), 9, dtype=torch.int32)
    rep = run_and_compare(ocfg, gcfg, draft, target, root, prefix, allow_diverged=B, allow_kinds=("cross_row_tie",))
    assert rep.status_bits & c2t.ST_INTERNAL == 0 and rep.status_bits == 0, rep.status_bits
print("debug-bounds cases ok")
"""


def test_parity_cases_under_index_checks():
    from paper_2502_13652_b200 import build
    lib = build.build(debug_bounds=True)
    env = dict(os.environ, C2T_LIBRARY=lib)
    code = CHILD.format(root=ROOT, tests=os.path.join(ROOT, "tests"))
    out = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=900)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    assert "debug-bounds cases ok" in out.stdout


GIVE_UP = r"""
import ctypes, sys, torch
sys.path.insert(0, {root!r}); sys.path.insert(0, {tests!r})
import paper_2502_13652_b200 as c2t
from parity_util import gen_inputs, make_configs, special_rows
assert c2t.LIB_PATH.endswith("libc2t_debug.so")
limit = ctypes.c_int.in_dll(c2t.lib(), "c2t_debug_task_wait_limit")
usual = limit.value
# rows shared by several CTAs and rows inside one; expand and prune in one launch, in two, with candidates set aside; the rows of a level
# streamed or in the registers of clusters, there also rows whose largest are found in rounds over all blocks
for B, V, F, dtype, M, kind in [(1, 32000, 4, torch.float32, 0, ""), (2, 70000, 8, torch.bfloat16, 0, ""), (5, 40000, 8, torch.float32, 0, ""),
                                (96, 4096, 10, torch.bfloat16, 0, ""), (6, 32000, 8, torch.bfloat16, 64, ""),
                                (2, 128256, 20, torch.bfloat16, 0, ""), (40, 40000, 8, torch.float32, 0, ""),
                                (3, 70000, 5, torch.float32, 0, "two_valued"), (6, 30000, 2, torch.bfloat16, 0, "two_valued")]:
    D, K, N = 4, 6, 20
    _, cfg = make_configs(B, V, D, K, F, N, 0.3 if not kind else 0.0, dtype, M=M)
    draft, target, root, prefix = gen_inputs(B, V, D, F, c2t.c2t_final_width(cfg), dtype)
    if kind:
        draft = [special_rows(kind, B, F, V, dtype) for _ in range(D)]
    draft = [t.cuda() for t in draft]; target = target.cuda(); root = root.cuda(); prefix = prefix.cuda()
    ctx = c2t.Context(cfg)

    def step(*limits):                                 # one per level
        ctx.c2t_begin_step(root, prefix)
        for l in range(D):
            limit.value = limits[l]
            ctx.c2t_expand_prune_level(l, draft[l])
        limit.value = usual
        ctx.c2t_prune(c2t.FINAL); ctx.c2t_build_verify(); ctx.c2t_accept(target)
        out = [v.cpu().clone() for v in list(ctx.verify.values()) + list(ctx.accepted.values())]
        return out, ctx.c2t_status()[1]

    out, status = step(0, usual, usual, usual)         # on a new workspace: every row of level 0 is given up
    assert all(s == c2t.ST_INTERNAL for s in status), status
    assert (out[0] == 1).all(), out[0]                 # the roots alone
    want, status = step(*[usual] * D)
    assert not any(status) and int(want[0].max()) > 1, status
    out, status = step(usual, usual, 0, usual)         # in the middle of a step
    assert all(s == c2t.ST_INTERNAL for s in status), status
    for few in ((usual, 1, 2, usual), (3, 8, 20, 50)):  # whatever runs out here
        step(*few)
    out, status = step(*[usual] * D)
    assert not any(status)
    for a, b in zip(out, want):
        assert torch.equal(a, b)
    ctx.close()
# levels of these shapes are in registers, one launch each; they stay there when the limit is changed
ctx = c2t.Context(make_configs(5, 40000, 4, 6, 8, 20, 0.3, torch.float32)[1])
x = torch.zeros(5, 8, 40000, device="cuda"); ints = torch.zeros(5, dtype=torch.int32, device="cuda")
for limit.value in (usual, 0):
    ctx.c2t_begin_step(ints, ints)
    n = ctx.c2t_launch_count()
    ctx.c2t_expand_prune_level(0, x)
    assert ctx.c2t_launch_count() == n + 1, limit.value
    assert all(s == (c2t.ST_INTERNAL if limit.value == 0 else 0) for s in ctx.c2t_status()[1])
ctx.close()
print("given-up rows ok")
"""


def test_a_wait_that_runs_out_ends_with_its_step():
    """Rows whose records do not come in time are reported as C2T_ST_INTERNAL, and the next step on the same workspace is right."""
    from paper_2502_13652_b200 import build
    env = dict(os.environ, C2T_LIBRARY=build.build(debug_bounds=True))
    code = GIVE_UP.format(root=ROOT, tests=os.path.join(ROOT, "tests"))
    out = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=900)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    assert "given-up rows ok" in out.stdout
