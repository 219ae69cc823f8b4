"""The host side of the library over a runtime that only writes down its calls (tests/fake_cuda.cpp): the order of clears, copies,
waits and launches, and what is left behind by a call that fails.  No GPU."""
import ctypes as C
import os
import subprocess

import pytest

import paper_2502_13652_b200 as c2t
from paper_2502_13652_b200 import binding

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")
STREAM = 0x77                                           # the caller's stream
LEGACY = 0x1                                            # cudaStreamLegacy


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fake") / "libc2t_fake.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-w", "-Wl,-Bsymbolic", "-I", os.path.join(CUDA, "include"), "-I",
                           os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2502_13652_b200", "csrc"), "-o", so,
                           os.path.join(ROOT, "tests", "fake_cuda.cpp")])
    L = C.CDLL(so)
    L.fake_log.restype = C.c_char_p
    L.c2t_workspace_bytes.restype = L.c2t_host_step_ints.restype = C.c_size_t
    L.fake_reset()
    return L


def config(B=3, V=4096, D=4, K=5, F=4, N=16, M=0, classifier=c2t.CLS_IDENTITY_JOINT, device=0):
    return binding.c2t_config(B, V, c2t.F32, D, K, F, N, 0.0, M, classifier, 0, None, None, None, None, 0, device)


def calls(L):
    return [line.split() for line in L.fake_log().decode().splitlines()]


class Ctx:
    def __init__(self, L, **kw):
        self.L, self.cfg = L, config(**kw)
        L.fake_reset()
        n = L.c2t_workspace_bytes(C.byref(self.cfg))
        self.mem = C.create_string_buffer(n + 512)
        base = (C.addressof(self.mem) + 255) & ~255
        self.h = C.c_void_p()
        assert L.c2t_init(C.byref(self.cfg), C.c_void_p(base), C.c_size_t(n), C.byref(self.h)) == c2t.OK

    def close(self):
        self.L.c2t_destroy(self.h)


def test_init_waits_for_its_clears(lib):
    """A first step may run on a stream that does not wait for the default one."""
    ctx = Ctx(lib)
    log = calls(lib)
    last = max(i for i, c in enumerate(log) if c[0] in ("memset", "memcpy"))
    assert ["sync", hex(LEGACY)] in log[last + 1:] or ["sync", "(nil)"] in log[last + 1:], log
    ctx.close()


def arg_max_calls(L, ctx, buf):
    keys, big = C.c_void_p(buf), C.c_int64(4096)
    h, s = ctx.h, C.c_void_p(STREAM)
    return {"accept": lambda: L.c2t_accept(h, keys, big, big, None, s),
            "argmax_shard": lambda: L.c2t_argmax_shard(h, keys, big, big, 4096, 0, keys, s),
            "lazy_argmax_shard": lambda: L.c2t_lazy_argmax_shard(h, keys, big, big, 4096, 0, keys, s)}


@pytest.mark.parametrize("second", ["accept", "argmax_shard", "lazy_argmax_shard"])
@pytest.mark.parametrize("first,kernel", [("accept", "accept_walk"), ("argmax_shard", "export_best"), ("lazy_argmax_shard", "export_lazy_best")])
def test_keys_of_an_arg_max_that_nobody_read(lib, first, kernel, second):
    """An arg-max pass takes the largest of what is there; if the launch that reads its keys failed, they must go before the next."""
    ctx = Ctx(lib)
    buf = (C.addressof(ctx.mem) + 255) & ~255
    assert lib.c2t_begin_step(ctx.h, C.c_void_p(buf), C.c_void_p(buf), C.c_void_p(STREAM)) == c2t.OK
    assert lib.c2t_prune(ctx.h, c2t.FINAL, None, C.c_void_p(STREAM)) == c2t.OK
    call = arg_max_calls(lib, ctx, buf)
    lib.fake_fail(kernel.encode(), 1)
    assert call[first]() == c2t.ECUDA
    lib.fake_reset()
    assert call[second]() == c2t.OK
    names = [c[0] for c in calls(lib)]
    assert names[:2] == ["memset_async", "argmax"], names
    lib.fake_reset()
    assert call[second]() == c2t.OK
    assert "memset_async" not in [c[0] for c in calls(lib)]           # once
    ctx.close()


def host_step(L, ctx, alias=None):
    """Issues a c2t_decode_step_host; returns its code and the staging ranges.  alias: bytes from the draft stage's start to the
    target stage's (default: apart)."""
    B, F, V, D = ctx.cfg.batch, ctx.cfg.frontier_cap, ctx.cfg.vocab, ctx.cfg.max_depth
    rows, tgt = B * F * V * 4, B * L.c2t_final_width(C.byref(ctx.cfg)) * V * 4
    draft = 0x10000000
    target = draft + (0x8000000 if alias is None else alias)
    ints = C.create_string_buffer(L.c2t_host_step_ints(C.byref(ctx.cfg)) * 4 + 64)
    host = C.create_string_buffer(64)
    at = (C.addressof(host) + 15) & ~15
    arr = (C.c_void_p * D)(*[at] * D)
    io = binding.c2t_host_step(arr, at, at, at, draft, target, (C.addressof(ints) + 15) & ~15, None, None, None, None, None)
    rc = L.c2t_decode_step_host(ctx.h, C.byref(io), C.c_void_p(STREAM))
    return rc, (draft, draft + rows), (target, target + tgt)


def races(log, stages):
    """Accesses to the staging buffers that nothing orders: (earlier, later) pairs of log lines.  A copy writes its range, a launch
    with a pointer reads the stage that begins there."""
    knows, events, touched, bad = {}, {}, [], []
    for i, c in enumerate(log):
        if c[0] == "record":
            events[c[1]] = set(knows.setdefault(c[2], set()))
        elif c[0] == "wait":
            knows.setdefault(c[1], set()).update(events.get(c[2], ()))
        elif c[0] == "copy" or (c[0] in ("expand", "argmax", "topm_entropy") and c[2] != "(nil)"):
            stream, lo = (c[3], int(c[1], 16)) if c[0] == "copy" else (c[1], int(c[2], 16))
            hi = lo + int(c[2]) if c[0] == "copy" else next((e for b, e in stages if b == lo), lo)
            mine = knows.setdefault(stream, set())
            for j, a, b, writes in touched:
                if a < hi and lo < b and (writes or c[0] == "copy") and j not in mine:
                    bad.append((log[j], c))
            touched.append((i, lo, hi, c[0] == "copy"))
            mine.add(i)
    return bad


@pytest.mark.parametrize("D", [1, 2, 4])
@pytest.mark.parametrize("N", [16, 3])
def test_host_step_leaves_its_rows_in_the_staging_buffers(lib, D, N):
    """The last level's rows in the one, all target rows in the other, and the arg-max of every node's row is taken."""
    ctx = Ctx(lib, D=D, N=N)
    lib.fake_reset()
    rc, draft, target = host_step(lib, ctx)
    assert rc == c2t.OK
    log = calls(lib)
    into = {hex(draft[0]): [], hex(target[0]): []}
    for c in log:
        if c[0] == "copy" and c[1] in into:
            into[c[1]].append(int(c[2]))
    assert into[hex(draft[0])][-1] == draft[1] - draft[0] and into[hex(target[0])][-1] == target[1] - target[0]
    assert [c[2] for c in log if c[0] == "argmax"] == [hex(target[0])]
    assert sum(c[0] == "expand" for c in log) == D
    assert not races(log, (draft, target))
    ctx.close()


@pytest.mark.parametrize("alias", [0, 4096, 16 * 3 * 4 * 4096, -4096])
def test_host_step_with_staging_buffers_that_overlap(lib, alias):
    """One buffer for both stages, or two that share a part: a copy must not meet the kernel that still reads there."""
    ctx = Ctx(lib)
    lib.fake_reset()
    rc, draft, target = host_step(lib, ctx, alias=alias)
    assert rc == c2t.OK
    assert not races(calls(lib), (draft, target))
    ctx.close()


@pytest.mark.parametrize("call,at", [("expand", 1), ("expand", 3), ("prune", 2), ("copy", 4), ("copy", 6), ("record", 3), ("wait", 4),
                                     ("final_prune", 1), ("argmax", 1), ("accept_walk", 1), ("sync", 1)])
def test_host_step_that_fails_waits_for_its_copies(lib, call, at):
    """The copies run on a stream that the caller does not have, from and to the caller's buffers."""
    ctx = Ctx(lib)
    assert host_step(lib, ctx)[0] == c2t.OK
    lib.fake_reset()
    lib.fake_fail(call.encode(), at)
    rc = host_step(lib, ctx)[0]
    assert rc == c2t.ECUDA
    log = calls(lib)
    own = {c[3] for c in log if c[0] == "copy"} - {hex(STREAM)}
    assert len(own) == 1
    last = max(i for i, c in enumerate(log) if c[0] == "copy" and c[3] in own)
    assert ["sync", own.pop()] in log[last + 1:], log
    lib.fake_reset()
    assert host_step(lib, ctx)[0] == c2t.OK             # and the context is still good
    ctx.close()


@pytest.mark.parametrize("fail", [None] + [("create_event", i) for i in range(1, 6)] + [("create_stream", 1)])
def test_host_step_makes_its_stream_once_on_the_device_of_the_context(lib, fail):
    """Whatever device is current, and however often making them fails."""
    ctx = Ctx(lib, device=2)
    lib.fake_reset()
    lib.cudaSetDevice(5)
    events, streams = lib.fake_events(), lib.fake_streams()
    if fail:
        lib.fake_fail(fail[0].encode(), fail[1])
        assert host_step(lib, ctx)[0] == c2t.ECUDA
        assert (lib.fake_events(), lib.fake_streams()) == (events, streams)
    for _ in range(2):
        assert host_step(lib, ctx)[0] == c2t.OK
    assert (lib.fake_events(), lib.fake_streams()) == (events + 5, streams + 1)
    made = [c for c in calls(lib) if c[0].startswith("create")]
    assert all(c[3] == "2" for c in made), made
    device = C.c_int()
    lib.cudaGetDevice(C.byref(device))
    assert device.value == 5
    ctx.close()
    assert (lib.fake_events(), lib.fake_streams()) == (events, streams)


def test_workspace_has_no_pool_where_nothing_is_set_aside(lib):
    """With M so large that the floors cannot hold M elements (here: more than a quarter of the row) the rows are read again."""
    def size(M):
        cfg = config(B=16, V=32768, F=8, M=M)
        return lib.c2t_workspace_bytes(C.byref(cfg))
    pool = 16 * 8 * 32768 * 4 // 48 * 16
    assert size(1000) - size(0) > pool
    assert size(12000) - size(0) < 4096
    ctx = Ctx(lib, M=2000)
    view = binding.c2t_view()
    assert lib.c2t_get_view(ctx.h, C.byref(view)) == c2t.OK and view.topm_from_pass
    ctx.close()


def device_step(L, ctx, **change):
    """Issues a c2t_decode_step; returns its code.  change: fields of the step; levels: {level: (pointer, seq_stride, row_stride)}."""
    D, V, B = ctx.cfg.max_depth, ctx.cfg.vocab, ctx.cfg.batch
    rows = [(0x20000000 + l * 0x100000, 4 * V, V) for l in range(D)]
    for l, r in change.pop("levels", {}).items():
        rows[l] = r
    pointers = (C.c_void_p * D)(*[r[0] for r in rows])
    strides = (C.c_int64 * (2 * D))(*[x for r in rows for x in r[1:]])
    step = binding.c2t_step(0x1000, 0x2000, pointers, strides, 0x30000000, 16 * V, V, None, None, None)
    for name, value in change.items():
        setattr(step, name, value)
    return L.c2t_decode_step(ctx.h, C.byref(step), C.c_void_p(STREAM))


LEVELS = ["expand", "prune"] * 4


@pytest.mark.parametrize("change,code,before", [
    (dict(draft_logits_dev=C.POINTER(C.c_void_p)()), c2t.EINVAL, []), (dict(draft_strides=C.POINTER(C.c_int64)()), c2t.EINVAL, []),
    (dict(root_tok_dev=None), c2t.EINVAL, []), (dict(prefix_len_dev=None), c2t.EINVAL, []),
    (dict(levels={0: (None, 16384, 4096)}), c2t.EINVAL, ["begin"]), (dict(levels={2: (None, 16384, 4096)}), c2t.EINVAL, ["begin"] + LEVELS[:4]),
    (dict(levels={2: (0x20000004, 16384, 4096)}), c2t.EALIGN, ["begin"] + LEVELS[:4]), (dict(levels={1: (0x20000000, 16386, 4096)}), c2t.EALIGN, ["begin"] + LEVELS[:2]),
    (dict(levels={1: (0x20000000, 16384, 4098)}), c2t.EALIGN, ["begin"] + LEVELS[:2]), (dict(levels={3: (0x20000000, 16384, 4092)}), c2t.EINVAL, ["begin"] + LEVELS[:6]),
    (dict(levels={3: (0x20000000, -16384, 4096)}), c2t.EINVAL, ["begin"] + LEVELS[:6]),
    (dict(target_logits_dev=None), c2t.EINVAL, ["begin"] + LEVELS + ["final_prune", "build_verify"]),
    (dict(target_logits_dev=0x30000008), c2t.EALIGN, ["begin"] + LEVELS + ["final_prune", "build_verify"]),
    (dict(target_row_stride=4092), c2t.EINVAL, ["begin"] + LEVELS + ["final_prune", "build_verify"]),
    (dict(), c2t.OK, ["begin"] + LEVELS + ["final_prune", "build_verify", "argmax", "accept_walk"])])
def test_device_step_stops_at_the_first_call_that_refuses(lib, change, code, before):
    """With the code of that call, after the launches of those before it; the next step is a whole one."""
    ctx = Ctx(lib)
    for what, want, names in ((dict(change), code, before), (dict(), c2t.OK, ["begin"] + LEVELS + ["final_prune", "build_verify", "argmax", "accept_walk"])):
        lib.fake_reset()
        assert device_step(lib, ctx, **what) == want
        assert [c[0] for c in calls(lib)] == names
    ctx.close()


def test_device_step_without_a_step_or_a_context(lib):
    ctx = Ctx(lib)
    assert lib.c2t_decode_step(ctx.h, None, None) == c2t.EINVAL and lib.c2t_decode_step(None, None, None) == c2t.EINVAL
    ctx.close()


class Rows:
    """As much of a CUDA tensor as a call's checks look at."""
    is_cuda, dtype = True, c2t.Config(1, 8).torch_dtype

    def __init__(self, *shape):
        self.shape = shape

    def dim(self):
        return len(self.shape)

    def stride(self, i=None):
        s = (self.shape[1] * self.shape[2], self.shape[2], 1)
        return s if i is None else s[i]

    def data_ptr(self):
        return 4096


def test_decode_step_launches_a_level_before_it_looks_at_the_next(monkeypatch):
    """The device has work while the rest is looked at, and a sequence of levels may run a draft model on the frontier emitted so far."""
    import torch
    log = []

    class Recorder:
        def __getattr__(self, name):
            return lambda *a: log.append((name,) + (tuple(a[1:2]) if "expand" in name or name == "c2t_prune" else ())) or 0

    class Levels:
        def __getitem__(self, level):
            log.append(("rows", level))
            return Rows(2, 4, 64)

    monkeypatch.setattr(binding, "lib", lambda: recorder)
    recorder = Recorder()
    ctx = object.__new__(binding.Context)
    ctx.cfg, ctx._h, ctx.B, ctx.D, ctx.V = c2t.Config(2, 64), None, 2, 3, 64
    ctx._frontier_c, ctx._verify_c, ctx._accept_c = binding.c2t_frontier(), binding.c2t_verify(), binding.c2t_accept_out()
    ints = Rows(1, 1, 2)
    ints.dtype, ints.numel = torch.int32, lambda: 2
    ctx.decode_step(Levels(), Rows(2, 5, 64), ints, ints, stream=0)
    assert log == [("c2t_begin_step",)] + [x for l in range(3) for x in (("rows", l), ("c2t_expand_prune_level", l))] + \
        [("c2t_prune", c2t.FINAL), ("c2t_build_verify",), ("c2t_accept",)]


@pytest.mark.parametrize("elem", [2, 4])
@pytest.mark.parametrize("K", [1, 4, 10, 16, 32])
def test_rows_in_registers_have_data_for_the_floor(lib, elem, K):
    """The floor is the K-th largest maximum of 64 groups of threads (or as many as there are warps).  Where fewer than K groups have data
    it is no floor at all, and where hardly more have most of the row may reach it: then the K largest are found in K rounds."""
    cluster, threads = C.c_int(), C.c_int()
    taken = set()
    for V in list(range(1, 3000, 53)) + [2003, 4000, 8000, 16000, 16384, 16385, 32000, 65536, 65537, 128256, 131072, 262144]:
        for rows in (1, 2, 3, 5, 9, 12, 18, 37, 74, 148, 296, 297):
            lib.fake_row_plan(V, elem, C.c_longlong(rows), K, 148, C.byref(cluster), C.byref(threads))
            if not cluster.value:
                continue
            taken.add(V)
            c, t = cluster.value, threads.value
            vectors = -(-V * elem // 16)
            part = -(-vectors // c)
            assert part <= 8 * t and rows * c * t <= 148 * 512
            groups = max(64, c * t // 32)
            width = c * t // groups                     # threads of a group
            with_data = sum(-(-min(t, max(0, min(part, vectors - r * part))) // width) for r in range(c))
            assert with_data >= min(groups, 1.5 * K), (V, rows, c, t, with_data)
    assert {4000, 16000, 32000, 65536} <= taken
