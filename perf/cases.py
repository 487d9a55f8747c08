"""The lineage path's workloads, for timing and for comparing outputs.

Every case is a source microbatch, or a step of one, as a program that keeps
its lineage on the GPU runs it: expand the parents, admit and reserve the
children in batches, commit their results as they arrive, assemble each
completed parent.  Inputs follow the distributions of the repository's five
configurations (tiny, document->page, video->clip->frame, extreme skew,
streaming), drawn on the GPU from the seed.  `prepare` holds what such a
program has before the pass: inputs and output arrays on the device, a context
with its streams and, where the program replays its wave loop, the captured
graph.  `run` is one pass through the public binding.

All outputs are whole numbers and bytes fixed by the lineage definitions, so
they are compared for equality (the CPU oracle under oracle/ computes each of
them; there is no rounding to state an error for).  Unsigned outputs are held
in signed tensors of the same width, assembled bytes in 64-bit words.
"""
import functools
import math

import numpy as np
import torch

import paper_2609_18703_gb300 as ro

PRESENT, FAILED = ro.RO_PRESENT, ro.RO_FAILED
DEV = "cuda"


def listed():
    return [
        # the smallest microbatch a service hands over: every call is launch and latency
        {"name": "tiny_1k", "kind": "pass", "fan": "tiny", "parents": 1000, "record": 64, "waves": 1,
         "batch": 64, "fail": 0.03, "streams": False, "graph": False},
        # an ordinary document->page microbatch, its results in a few arrivals
        {"name": "docs_50k", "kind": "pass", "fan": "docpage", "parents": 50_000, "record": 0, "waves": 4,
         "batch": 256, "fail": 0.05, "streams": True, "graph": False},
        # the benchmark's document->page level: 256 arrival waves, the wave loop replayed as a graph
        {"name": "docs_1m", "kind": "pass", "fan": "docpage", "parents": 1_000_000, "record": 0, "waves": 256,
         "batch": 256, "fail": 0.05, "streams": True, "graph": True},
        # extreme fan-out skew: 110 million 32-byte children, 91 % of them under 1,000 parents
        {"name": "skew_10m", "kind": "pass", "fan": "skew", "parents": 10_000_000, "record": 32, "waves": 1,
         "batch": 256, "fail": 0.0, "streams": True, "graph": False},
        # payloads in pinned host memory, read and written in place by the copy
        {"name": "host_10k", "kind": "pass", "fan": "docpage", "parents": 10_007, "record": 0, "waves": 4,
         "batch": 256, "fail": 0.05, "streams": True, "graph": False, "host": True},
        # F.filter before each commit, list-structured output, then a re-read of parents in the caller's order
        {"name": "lists_60k", "kind": "pass", "fan": "docpage", "parents": 60_001, "record": 0, "waves": 8,
         "batch": 256, "fail": 0.01, "streams": True, "graph": True, "drop": 0.1, "lists": True},
        # video->clip->frame: one level's assembly committed as the reports of the level above
        {"name": "video_100k", "kind": "nested", "parents": 100_000, "record": 512, "batch": 1024},
        # four Calls, children ready in waves, reserved in whole batches, results back in the same wave
        {"name": "stream_10m", "kind": "stream", "children": 10_000_000, "record": 1024, "waves": 200,
         "batch": 256, "calls": 4, "fail": 0.02},
        # parent-bound reservation of pages in readiness order
        {"name": "bound_250k", "kind": "bound", "parents": 250_000, "waves": 2, "batch": 256},
        # a failed attempt of many batches goes back to its recovery queue and is dispatched again
        {"name": "retry_250k", "kind": "retry", "parents": 250_000, "batch": 256, "batches": 512},
        # an unreliable executor: repeated and stale reports, typed group failures
        {"name": "faults_100k", "kind": "faults", "parents": 100_000, "record": 512, "waves": 16, "batch": 256,
         "repeats": 0.01, "poisoned": 20},
        # the expansion for callers that cannot allocate
        {"name": "noalloc_1m", "kind": "noalloc", "parents": 1_000_000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tiny", "docs", "docs", "skew", "host", "lists", "nested", "stream", "bound", "retry",
                       "faults", "noalloc"])
    batch = rng.choice([32, 64, 100, 256, 1024, 2048])
    if kind == "tiny":
        return {"kind": "pass", "fan": "tiny", "parents": _log(rng, 500, 20_000), "record": _log(rng, 16, 512),
                "waves": rng.randint(1, 2), "batch": batch, "fail": round(rng.uniform(0, 0.1), 3),
                "streams": False, "graph": False}
    if kind == "docs":
        waves = _log(rng, 1, 256)
        return {"kind": "pass", "fan": "docpage", "parents": _log(rng, 2_000, 700_000), "record": 0,
                "waves": waves, "batch": batch, "fail": round(rng.uniform(0, 0.08), 3), "streams": True,
                "graph": waves > 6}
    if kind == "skew":
        return {"kind": "pass", "fan": "skew", "parents": _log(rng, 40_000, 6_000_000),
                "record": rng.choice([17, 32, 32, 48, 100]), "waves": rng.randint(1, 3), "batch": batch,
                "fail": 0.0, "streams": True, "graph": False}
    if kind == "host":
        return {"kind": "pass", "fan": "docpage", "parents": _log(rng, 1_000, 12_000), "record": 0,
                "waves": rng.randint(1, 6), "batch": batch, "fail": round(rng.uniform(0, 0.08), 3),
                "streams": True, "graph": False, "host": True}
    if kind == "lists":
        waves = _log(rng, 2, 24)
        return {"kind": "pass", "fan": "docpage", "parents": _log(rng, 2_000, 120_000), "record": 0,
                "waves": waves, "batch": batch, "fail": round(rng.uniform(0, 0.02), 3), "streams": True,
                "graph": waves > 6, "drop": round(rng.uniform(0.02, 0.5), 3), "lists": True}
    if kind == "nested":
        return {"kind": "nested", "parents": _log(rng, 1_000, 100_000), "record": _log(rng, 64, 512), "batch": batch}
    if kind == "stream":
        waves = _log(rng, 8, 200)
        return {"kind": "stream", "children": waves * _log(rng, 2_000, 50_000), "record": _log(rng, 64, 1024),
                "waves": waves, "batch": batch, "calls": rng.randint(1, 4), "fail": round(rng.uniform(0, 0.05), 3)}
    if kind == "bound":
        return {"kind": "bound", "parents": _log(rng, 1_000, 500_000), "waves": rng.randint(1, 4), "batch": batch}
    if kind == "retry":
        return {"kind": "retry", "parents": _log(rng, 10_000, 500_000), "batch": batch,
                "batches": _log(rng, 1, 64_000 // batch)}
    if kind == "faults":
        return {"kind": "faults", "parents": _log(rng, 2_000, 150_000), "record": _log(rng, 64, 512),
                "waves": rng.randint(4, 24), "batch": batch, "repeats": round(rng.uniform(0, 0.03), 4),
                "poisoned": rng.randint(0, 40)}
    return {"kind": "noalloc", "parents": _log(rng, 1_000, 4_000_000)}


# ---------------------------------------------------------------------------- inputs
class State:
    """What a program keeps between passes.  Its context goes with it."""
    ctx = None
    graph = None

    def __del__(self):
        self.graph = None
        if self.ctx:
            ro.ro_ctx_destroy(self.ctx)
            self.ctx = None


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _lognormal(g, n, mu, sigma, lo, hi):
    x = torch.empty(n, dtype=torch.float64, device=DEV).log_normal_(mu, sigma, generator=g)
    return x.round_().clamp_(lo, hi).to(torch.int64)


FANS = {"tiny": (2.0, 1.0, 1, 500), "docpage": (2.3, 1.0, 1, 2000), "stream": (2.5, 1.2, 0, 1 << 20)}


# Sizes (children per parent, bytes per record) are one draw of their
# distribution, dealt out by the seed: inputs of another seed differ, the
# arrays' lengths do not.
def _deal(g, x):
    return x[torch.randperm(x.numel(), generator=g, device=DEV)]


def _counts(g, fan, parents):
    if fan == "skew":   # one child each, but for one parent in 10,000 with 100,000 (fewer when the case is small)
        heavy, size = _skew(parents)
        c = torch.ones(parents, dtype=torch.int64, device=DEV)
        c[:heavy] = size
    else:
        c = _lognormal(_gen(1), parents, *FANS[fan])
    return _deal(g, c)


def _skew(parents):
    return max(1, parents // 10_000), min(100_000, max(5_000, parents // 10))


def _lengths(g, n, record):
    if record:
        return torch.full((n,), record, dtype=torch.int64, device=DEV)
    return _deal(g, _lognormal(_gen(2), n, 7.5, 0.8, 256, 65536))   # page payloads


def _out_cap(case, total, gathered):
    """Output capacity: all records, or for a large pass a little over what its assembled parents should hold."""
    fan, fail = case.get("fan", "stream"), case["fail"]
    keep = 1.0 if fan == "skew" else _expected(fan, fail, case["record"])[2]
    cap = min(total, int(1.05 * keep * total) + (64 << 20)) + 16
    assert gathered + 16 <= cap
    return cap


def _bytes(g, n):
    """n random bytes (a multiple of 16 allocated), as the executors' result arena."""
    words = torch.empty(n // 8 + 4, dtype=torch.int64, device=DEV)
    return words.random_(generator=g).view(torch.uint8)


def _zeros(n, dtype):
    return torch.zeros(max(int(n), 1), dtype=dtype, device=DEV)


def _bounds(n, waves):
    sizes = np.full(waves, n // waves, dtype=np.int64)
    sizes[: n % waves] += 1
    return [int(x) for x in np.concatenate([[0], np.cumsum(sizes)])]


def _parents_of(counts):
    return torch.repeat_interleave(torch.arange(counts.numel(), device=DEV), counts)


def _excl(x):
    return torch.cumsum(x, 0) - x


def _expand_bufs(s, counts):
    s.P, s.N = counts.numel(), int(counts.sum())
    s.counts = counts.to(torch.int32)
    s.offsets = _zeros(s.P + 1, torch.int64)
    s.parents, s.ordinals = _zeros(s.N, torch.int32), _zeros(s.N, torch.int32)
    s.empties = _zeros(s.P, torch.int32)


def _context(s, calls=1, streams=True):
    s.stream = torch.cuda.Stream()
    s.ctx = ro.ro_ctx_create(torch.cuda.current_device(), s.stream, calls)
    if streams:
        s.side = (torch.cuda.Stream(), torch.cuda.Stream())
        ro.ro_ctx_set_streams(s.ctx, *s.side)


def _check(s, status):
    if status != ro.RO_OK:
        raise ro.RoError("pass", status, ro.ro_last_error(s.ctx))


def _at(t, i):
    """The address of entry i of a tensor (a wave's window of an array)."""
    return t.data_ptr() + i * t.element_size()


def _expand(s):
    st, n, _, xid = ro.ro_expand(s.ctx, -1, s.counts, s.P, s.calls_of, s.offsets, s.parents, s.ordinals, s.N,
                                 s.empties)
    _check(s, st)
    return xid


def _capture(s, loop):
    """Run the wave loop once (it sizes the context's buffers), then capture it for replay."""
    ro.ro_ctx_reset(s.ctx)
    with torch.cuda.stream(s.stream):
        loop(s, _expand(s))
    _check(s, ro.ro_ctx_sync(s.ctx))
    ro.ro_ctx_reset(s.ctx)
    xid = _expand(s)
    s.graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(s.graph, stream=s.stream):
        loop(s, xid)


def _run_waves(s, loop):
    ro.ro_ctx_reset(s.ctx)
    with torch.cuda.stream(s.stream):
        xid = _expand(s)
        if s.graph is not None:
            s.graph.replay()
        else:
            loop(s, xid)


# ---------------------------------------------------------------------------- one level, whole pass
def _prepare_pass(case, seed):
    s, g = State(), _gen(seed)
    counts = _counts(g, case["fan"], case["parents"])
    _expand_bufs(s, counts)
    s.calls_of = None
    s.bounds = _bounds(s.N, case["waves"])
    W = case["waves"]
    # reports in arrival order, their payloads packed back to back in that order
    child = torch.randperm(s.N, generator=g, device=DEV)
    failed = torch.rand(s.N, generator=g, device=DEV) < case["fail"]
    length = _lengths(g, s.N, case["record"])
    total = int(length.sum())
    length[failed] = 0
    off = _excl(length)
    s.arena_bytes = int(length.sum())
    state = torch.where(failed, FAILED, PRESENT).to(torch.uint8)
    s.child, s.state, s.len, s.off = child.to(torch.int32), state, length.to(torch.int32), off
    par = _parents_of(counts)[child]
    bad = torch.zeros(s.P, dtype=torch.bool, device=DEV)
    bad[par[failed]] = True
    s.out_cap = _out_cap(case, total, int(length[~bad[par]].sum()))
    s.keep = s.arrived = None
    if case.get("drop"):
        s.keep = (torch.rand(s.N, generator=g, device=DEV) >= case["drop"]).to(torch.uint8)
        s.arrived = state.clone()   # what the executors report, before the predicate
    s.lists = bool(case.get("lists"))
    if s.lists:   # a window of entries per wave, as many as the parents it completes have members
        wave = torch.repeat_interleave(torch.arange(W, device=DEV), torch.tensor(np.diff(s.bounds), device=DEV))
        last = torch.zeros(s.P, dtype=torch.int64, device=DEV).scatter_reduce_(0, par, wave, "amax")
        entries = torch.bincount(last, weights=counts.double(), minlength=W).long().tolist()
        s.entry_cap, s.entry_at = entries, np.concatenate([[0], np.cumsum(entries)]).tolist()
        s.elem_base, s.elem_state = _zeros(s.N + W, torch.int64), _zeros(s.N, torch.uint8)
        s.elem_off, s.elem_len, s.n_elems = _zeros(s.N, torch.int64), _zeros(s.N, torch.int32), _zeros(W, torch.int64)
        # parents read again, in an order of the caller's
        s.again = torch.randperm(s.P, generator=g, device=DEV)[: s.P // 2].to(torch.int32)
        n = s.again.numel()
        s.again_status, s.again_off = _zeros(n, torch.uint8), _zeros(n + 1, torch.int64)
    del par, failed, length, off, child
    s.arena = _bytes(g, s.arena_bytes)
    s.out = _zeros(s.out_cap // 8 + 1, torch.int64)
    if s.lists:
        s.again_out = torch.zeros_like(s.out)
    if case.get("host"):
        s.arena = s.arena.cpu().pin_memory()
        s.out = s.out.cpu().pin_memory()
    s.batch = case["batch"]
    s.batched, s.n_batched = _zeros(s.N, torch.int32), _zeros(1, torch.int64)
    s.code, s.done, s.n_done = _zeros(s.N, torch.uint8), _zeros(s.N, torch.int32), _zeros(W, torch.int64)
    s.status, s.out_off, s.out_len = _zeros(s.N, torch.uint8), _zeros(s.N + W, torch.int64), _zeros(s.N, torch.int32)
    s.cursor, s.out_bytes = _zeros(1, torch.int64), _zeros(W, torch.int64)
    torch.cuda.synchronize()
    _context(s, streams=case["streams"])
    if case["graph"]:
        _capture(s, _waves_pass)
    return s


def _waves_pass(s, xid):
    st, _, _ = ro.ro_batch_ready(s.ctx, xid, 0, None, 0, s.batch, True, s.batched, s.N, s.n_batched, want_host=False)
    _check(s, st)
    s.cursor.zero_()
    if s.arrived is not None:
        s.state.copy_(s.arrived)
    for w in range(len(s.bounds) - 1):
        a, b = s.bounds[w], s.bounds[w + 1]
        n = b - a
        k = min(n, s.P)   # parents the wave can complete
        if s.keep is not None:
            _check(s, ro.ro_filter_reports(s.ctx, _at(s.state, a), _at(s.keep, a), n))
        st, _ = ro.ro_gather_commit(s.ctx, xid, n, None, _at(s.child, a), _at(s.state, a), _at(s.len, a),
                                    _at(s.off, a), None, s.arena_bytes, _at(s.code, a), _at(s.done, a), k,
                                    _at(s.n_done, w), want_host=False)
        _check(s, st)
        if s.lists:
            e = s.entry_at[w]
            st, _, _ = ro.ro_assemble_list(
                s.ctx, xid, s.arena, s.arena_bytes, None, k, None, _at(s.status, a), _at(s.out_off, a + w),
                _at(s.out_len, a), s.out, s.out_cap, s.cursor, _at(s.out_bytes, w), _at(s.elem_base, a + w),
                _at(s.elem_state, min(e, s.N - 1)), _at(s.elem_off, min(e, s.N - 1)), _at(s.elem_len, min(e, s.N - 1)),
                s.entry_cap[w], _at(s.n_elems, w), want_host=False)
        else:
            st, _ = ro.ro_assemble(s.ctx, xid, s.arena, s.arena_bytes, None, k, None, _at(s.status, a),
                                   _at(s.out_off, a + w), _at(s.out_len, a), s.out, s.out_cap, s.cursor,
                                   _at(s.out_bytes, w), want_host=False)
        _check(s, st)
    if s.lists:
        st, _ = ro.ro_assemble(s.ctx, xid, s.arena, s.arena_bytes, s.again, s.again.numel(), None, s.again_status,
                               s.again_off, None, s.again_out, s.out_cap, want_host=False)
        _check(s, st)
    ro.ro_ctx_join(s.ctx)


def _run_pass(s):
    _run_waves(s, _waves_pass)
    out = {"offsets": s.offsets, "parents": s.parents, "ordinals": s.ordinals, "batched": s.batched,
           "n_batched": s.n_batched, "code": s.code, "done": s.done, "n_done": s.n_done, "status": s.status,
           "out_off": s.out_off, "out_len": s.out_len, "out_bytes": s.out_bytes, "out": s.out}
    if s.lists:
        out.update(state=s.state, elem_base=s.elem_base, elem_state=s.elem_state, elem_off=s.elem_off,
                   elem_len=s.elem_len, n_elems=s.n_elems, again_status=s.again_status, again_off=s.again_off,
                   again_out=s.again_out)
    return out


# ---------------------------------------------------------------------------- nested levels
def _prepare_nested(case, seed):
    s, g = State(), _gen(seed)
    u = 1.0 - torch.rand(case["parents"], generator=_gen(3), device=DEV, dtype=torch.float64)
    clips = _deal(g, torch.clamp(torch.floor(u ** (-1.0 / 1.5)), max=1000).to(torch.int64))
    C = int(clips.sum())
    frames = _deal(g, torch.randint(8, 65, (C,), generator=_gen(4), device=DEV))
    F = int(frames.sum())
    s.V, s.C, s.F, s.batch = case["parents"], C, F, case["batch"]
    s.clips, s.frames = clips.to(torch.int32), frames.to(torch.int32)
    child = torch.randperm(F, generator=g, device=DEV)
    s.child = child.to(torch.int32)
    s.state = torch.full((F,), PRESENT, dtype=torch.uint8, device=DEV)
    s.len = torch.full((F,), case["record"], dtype=torch.int32, device=DEV)
    s.off = torch.arange(F, device=DEV) * case["record"]
    s.bytes = F * case["record"]
    s.arena = _bytes(g, s.bytes)
    s.off1, s.par1, s.ord1 = _zeros(s.V + 1, torch.int64), _zeros(C, torch.int32), _zeros(C, torch.int32)
    s.off2, s.par2, s.ord2 = _zeros(C + 1, torch.int64), _zeros(F, torch.int32), _zeros(F, torch.int32)
    s.bat1, s.bat2 = _zeros(C, torch.int32), _zeros(F, torch.int32)
    s.code1, s.code2 = _zeros(C, torch.uint8), _zeros(F, torch.uint8)
    s.done1, s.done2, s.n_done = _zeros(s.V, torch.int32), _zeros(C, torch.int32), _zeros(2, torch.int64)
    s.status1, s.status2 = _zeros(s.V, torch.uint8), _zeros(C, torch.uint8)
    s.oo1, s.oo2 = _zeros(s.V + 1, torch.int64), _zeros(C + 1, torch.int64)
    s.ol1, s.ol2 = _zeros(s.V, torch.int32), _zeros(C, torch.int32)
    s.out1, s.out2 = _zeros(s.bytes // 8 + 3, torch.int64), _zeros(s.bytes // 8 + 3, torch.int64)
    torch.cuda.synchronize()
    _context(s)
    return s


def _run_nested(s):
    cap = s.bytes + 16
    ro.ro_ctx_reset(s.ctx)
    st, _, _, x1 = ro.ro_expand(s.ctx, -1, s.clips, s.V, None, s.off1, s.par1, s.ord1, s.C)
    _check(s, st)
    st, _, _, x2 = ro.ro_expand(s.ctx, x1, s.frames, s.C, None, s.off2, s.par2, s.ord2, s.F)
    _check(s, st)
    for x, b, n in ((x2, s.bat2, s.F), (x1, s.bat1, s.C)):
        _check(s, ro.ro_batch_ready(s.ctx, x, 0, None, 0, s.batch, True, b, n, None, want_host=False)[0])
    st, _ = ro.ro_gather_commit(s.ctx, x2, s.F, None, s.child, s.state, s.len, s.off, None, s.bytes, s.code2,
                                s.done2, s.C, _at(s.n_done, 1), want_host=False)
    _check(s, st)
    st, _ = ro.ro_assemble(s.ctx, x2, s.arena, s.bytes, None, s.C, None, s.status2, s.oo2, s.ol2, s.out2, cap,
                           want_host=False)
    _check(s, st)
    ro.ro_ctx_join(s.ctx)   # the clips' reports are the assembly's outputs
    st, _ = ro.ro_gather_commit(s.ctx, x1, s.C, None, s.done2, s.status2, s.ol2, s.oo2, None, s.bytes, s.code1,
                                s.done1, s.V, s.n_done, want_host=False)
    _check(s, st)
    st, _ = ro.ro_assemble(s.ctx, x1, s.out2.view(torch.uint8), s.bytes, None, s.V, None, s.status1, s.oo1, s.ol1,
                           s.out1, cap, want_host=False)
    _check(s, st)
    ro.ro_ctx_join(s.ctx)
    return {k: getattr(s, k) for k in ("off1", "par1", "ord1", "off2", "par2", "ord2", "bat1", "bat2", "code1", "code2",
                                       "done1", "done2", "n_done", "status1", "status2", "oo1", "oo2", "ol1", "ol2",
                                       "out1", "out2")}


# ---------------------------------------------------------------------------- several Calls, streaming
def _prepare_stream(case, seed):
    s, g = State(), _gen(seed)
    W, B, K = case["waves"], case["batch"], case["calls"]
    parents = max(1, int(case["children"] / math.exp(2.5 + 0.72)))
    counts = _counts(g, "stream", parents)
    _expand_bufs(s, counts)
    s.calls_of = (torch.arange(parents, device=DEV) % K).to(torch.uint8)
    par = _parents_of(counts)
    ready = torch.randperm(s.N, generator=g, device=DEV)
    s.bounds, s.W, s.B, s.K = _bounds(s.N, W), W, B, K
    s.cand = ready.to(torch.int32)
    failed = torch.rand(s.N, generator=g, device=DEV) < case["fail"]
    length = torch.where(failed, 0, case["record"])
    off = _excl(length)   # records lie in child order
    s.arena_bytes = int(length.sum())
    bad = torch.zeros(parents, dtype=torch.bool, device=DEV)
    bad[par[failed]] = True
    s.out_cap = _out_cap(case, s.N * case["record"], int(length[~bad[par]].sum()))
    # which children each wave reserves (whole batches; everything with the last), in random arrival order
    call_of = s.calls_of.long()[par[ready]]
    wave_of = torch.repeat_interleave(torch.arange(W, device=DEV), torch.tensor(np.diff(s.bounds), device=DEV))
    s.taken, order, at = [], [], []
    for k in range(K):
        mine = call_of == k
        queue = ready[mine]
        ends = torch.cumsum(torch.bincount(wave_of[mine], minlength=W), 0).cpu().numpy()
        upto = ends // B * B
        upto[-1] = ends[-1]
        s.taken.append([0] + [int(x) for x in upto])
        order.append(queue)
        at.append(torch.repeat_interleave(torch.arange(W, device=DEV),
                                          torch.tensor(np.diff(np.concatenate([[0], upto])), device=DEV)))
    order, at = torch.cat(order), torch.cat(at)
    mix = torch.randperm(s.N, generator=g, device=DEV)
    order, at = order[mix], at[mix]
    at, idx = torch.sort(at, stable=True)
    child = order[idx]
    s.reports = [0] + torch.cumsum(torch.bincount(at, minlength=W), 0).tolist()
    s.child, s.off = child.to(torch.int32), off[child]
    s.state = torch.where(failed, FAILED, PRESENT).to(torch.uint8)[child]
    s.len = length[child].to(torch.int32)
    del par, ready, failed, length, off, call_of, wave_of, order, at, mix, idx, child
    s.arena = _bytes(g, s.arena_bytes)
    s.out = _zeros(s.out_cap // 8 + 1, torch.int64)
    s.batched = [_zeros(s.N, torch.int32) for k in range(K)]
    s.n_batched = _zeros(W * K, torch.int64)
    s.code, s.done, s.n_done = _zeros(s.N, torch.uint8), _zeros(s.N, torch.int32), _zeros(W, torch.int64)
    s.status, s.out_off, s.out_len = _zeros(s.N, torch.uint8), _zeros(s.N + W, torch.int64), _zeros(s.N, torch.int32)
    s.cursor = _zeros(1, torch.int64)
    torch.cuda.synchronize()
    _context(s, calls=K)
    _capture(s, _waves_stream)
    return s


def _waves_stream(s, xid):
    s.cursor.zero_()
    for w in range(s.W):
        a, b = s.bounds[w], s.bounds[w + 1]
        bufs = [s.batched[k].data_ptr() + 4 * s.taken[k][w] for k in range(s.K)]
        caps = [s.taken[k][-1] - s.taken[k][w] for k in range(s.K)]
        _check(s, ro.ro_batch_ready_calls(s.ctx, xid, list(range(s.K)), _at(s.cand, a), b - a, s.B, w == s.W - 1, bufs,
                                          caps, [_at(s.n_batched, w * s.K + k) for k in range(s.K)]))
        a, b = s.reports[w], s.reports[w + 1]
        k = min(b - a, s.P)
        if b == a:   # no whole batch yet
            continue
        st, _ = ro.ro_gather_commit(s.ctx, xid, b - a, None, _at(s.child, a), _at(s.state, a), _at(s.len, a),
                                    _at(s.off, a), None, s.arena_bytes, _at(s.code, a), _at(s.done, a), k,
                                    _at(s.n_done, w), want_host=False)
        _check(s, st)
        st, _ = ro.ro_assemble(s.ctx, xid, s.arena, s.arena_bytes, None, k, None, _at(s.status, a),
                               _at(s.out_off, a + w), _at(s.out_len, a), s.out, s.out_cap, s.cursor, None,
                               want_host=False)
        _check(s, st)
    ro.ro_ctx_join(s.ctx)


def _run_stream(s):
    _run_waves(s, _waves_stream)
    return {"offsets": s.offsets, "parents": s.parents, "ordinals": s.ordinals, "empties": s.empties,
            "batched": s.batched, "n_batched": s.n_batched, "code": s.code, "done": s.done, "n_done": s.n_done,
            "status": s.status, "out_off": s.out_off, "out_len": s.out_len, "out": s.out}


# ---------------------------------------------------------------------------- parent-bound reservation
def _prepare_bound(case, seed):
    s, g = State(), _gen(seed)
    _expand_bufs(s, _counts(g, "docpage", case["parents"]))
    s.calls_of, s.batch, W = None, case["batch"], case["waves"]
    s.bounds = _bounds(s.N, W)
    s.cand = torch.randperm(s.N, generator=g, device=DEV).to(torch.int32)
    s.batched, s.batch_off = _zeros(s.N, torch.int32), _zeros(s.N + W, torch.int64)
    s.n_batched, s.n_batches = _zeros(W, torch.int64), _zeros(W, torch.int64)
    torch.cuda.synchronize()
    _context(s, streams=False)
    return s


def _run_bound(s):
    ro.ro_ctx_reset(s.ctx)
    xid = _expand(s)
    for w in range(len(s.bounds) - 1):
        a, b = s.bounds[w], s.bounds[w + 1]
        st, _, _ = ro.ro_batch_ready_parent(s.ctx, xid, 0, _at(s.cand, a), b - a, s.batch, True,
                                            _at(s.batched, a), b - a, _at(s.batch_off, a + w), b - a + 1,
                                            _at(s.n_batched, w), _at(s.n_batches, w), want_host=False)
        _check(s, st)
    return {"offsets": s.offsets, "parents": s.parents, "ordinals": s.ordinals, "batched": s.batched,
            "batch_off": s.batch_off, "n_batched": s.n_batched, "n_batches": s.n_batches}


# ---------------------------------------------------------------------------- retry
def _prepare_retry(case, seed):
    s, g = State(), _gen(seed)
    _expand_bufs(s, _counts(g, "docpage", case["parents"]))
    s.calls_of, s.batch = None, case["batch"]
    n = min(s.N, case["batches"] * case["batch"])
    s.failed = torch.randperm(s.N, generator=g, device=DEV)[:n].to(torch.int32)
    s.batched, s.n_batched = _zeros(s.N, torch.int32), _zeros(1, torch.int64)
    s.again, s.n_again = _zeros(n, torch.int32), _zeros(1, torch.int64)
    torch.cuda.synchronize()
    _context(s, streams=False)
    s.xid = _expand(s)   # every child is dispatched
    st, nb, _ = ro.ro_batch_ready(s.ctx, s.xid, 0, None, 0, s.batch, True, s.batched, s.N, s.n_batched)
    _check(s, st)
    return s


def _run_retry(s):
    st, _ = ro.ro_retry(s.ctx, s.xid, 0, s.failed, s.failed.numel(), want_host=False)
    _check(s, st)
    st, _, _ = ro.ro_batch_ready(s.ctx, s.xid, 0, s.failed, 0, s.batch, True, s.again, s.again.numel(), s.n_again,
                                 want_host=False)
    _check(s, st)
    return {"again": s.again, "n_again": s.n_again}


# ---------------------------------------------------------------------------- an unreliable executor
def _prepare_faults(case, seed):
    s, g = State(), _gen(seed)
    counts = _counts(g, "docpage", case["parents"])
    _expand_bufs(s, counts)
    W = case["waves"]
    s.calls_of, s.batch, s.W = None, case["batch"], W
    s.bounds = _bounds(s.N, W)
    ready = torch.randperm(s.N, generator=g, device=DEV)
    s.cand = ready.to(torch.int32)
    R = case["record"]
    s.arena_bytes = s.N * R
    state = torch.full((s.N,), PRESENT, dtype=torch.uint8, device=DEV)
    big = torch.argsort(counts, descending=True)[: case["poisoned"]]
    state[_excl(counts)[big]] = ro.RO_GROUP_FAILURE   # the first page of each poisoned document
    # per wave: the wave's reports, then repeats of some of them in random places, then stale ones (wrong generation)
    parts, gens, s.at = [], [], [0]
    for w in range(W):
        mine = ready[s.bounds[w]:s.bounds[w + 1]]
        extra = int(case["repeats"] * mine.numel())
        pick = torch.randint(0, mine.numel(), (2 * extra,), generator=g, device=DEV)
        ch = torch.cat([mine, mine[pick]])
        gen = torch.zeros(ch.numel(), dtype=torch.int32, device=DEV)
        gen[mine.numel() + extra:] = 1
        mix = torch.randperm(ch.numel(), generator=g, device=DEV)
        parts.append(ch[mix])
        gens.append(gen[mix])
        s.at.append(s.at[-1] + ch.numel())
    child = torch.cat(parts)
    s.child, s.gen, s.state, s.off = child.to(torch.int32), torch.cat(gens), state[child], child * R
    s.len = torch.full((child.numel(),), R, dtype=torch.int32, device=DEV)
    s.arena = _bytes(g, s.arena_bytes)
    s.out_cap = s.arena_bytes + 16
    s.out = _zeros(s.out_cap // 8 + 1, torch.int64)
    n = child.numel()
    s.batched, s.n_batched = _zeros(s.N, torch.int32), _zeros(W, torch.int64)
    s.code, s.done, s.n_done = _zeros(n, torch.uint8), _zeros(n, torch.int32), _zeros(W, torch.int64)
    s.status, s.out_off = _zeros(n, torch.uint8), _zeros(n + W, torch.int64)
    s.cursor = _zeros(1, torch.int64)
    torch.cuda.synchronize()
    _context(s)
    return s


def _waves_faults(s, xid):
    s.cursor.zero_()
    for w in range(s.W):
        a, b = s.bounds[w], s.bounds[w + 1]
        st, _, _ = ro.ro_batch_ready(s.ctx, xid, 0, _at(s.cand, a), b - a, s.batch, True,
                                     _at(s.batched, a), b - a, _at(s.n_batched, w), want_host=False)
        _check(s, st)
        a, b = s.at[w], s.at[w + 1]
        k = min(b - a, s.P)
        st, _ = ro.ro_gather_commit(s.ctx, xid, b - a, None, _at(s.child, a), _at(s.state, a), _at(s.len, a),
                                    _at(s.off, a), _at(s.gen, a), s.arena_bytes, _at(s.code, a), _at(s.done, a), k,
                                    _at(s.n_done, w), want_host=False)
        _check(s, st)
        st, _ = ro.ro_assemble(s.ctx, xid, s.arena, s.arena_bytes, None, k, None, _at(s.status, a),
                               _at(s.out_off, a + w), None, s.out, s.out_cap, s.cursor, None, want_host=False)
        _check(s, st)
    ro.ro_ctx_join(s.ctx)


def _run_faults(s):
    _run_waves(s, _waves_faults)
    return {"batched": s.batched, "n_batched": s.n_batched, "code": s.code, "done": s.done, "n_done": s.n_done,
            "status": s.status, "out_off": s.out_off, "out": s.out}


# ---------------------------------------------------------------------------- allocation-free expansion
def _prepare_noalloc(case, seed):
    s, g = State(), _gen(seed)
    _expand_bufs(s, _counts(g, "docpage", case["parents"]))
    s.stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    return s


def _run_noalloc(s):
    st, n, e = ro.ro_expand_noalloc(s.counts, s.P, s.offsets, s.parents, s.ordinals, s.N, s.empties, s.stream)
    if st != ro.RO_OK:
        raise ro.RoError("ro_expand_noalloc", st)
    return {"offsets": s.offsets, "parents": s.parents, "ordinals": s.ordinals, "n": n, "n_empty": e}


# ---------------------------------------------------------------------------- the interface
PREPARE = {"pass": _prepare_pass, "nested": _prepare_nested, "stream": _prepare_stream, "bound": _prepare_bound,
           "retry": _prepare_retry, "faults": _prepare_faults, "noalloc": _prepare_noalloc}
RUN = {"pass": _run_pass, "nested": _run_nested, "stream": _run_stream, "bound": _run_bound, "retry": _run_retry,
       "faults": _run_faults, "noalloc": _run_noalloc}


def prepare(case, seed):
    s = PREPARE[case["kind"]](case, seed)
    s.kind = case["kind"]
    return s


def run(state):
    return RUN[state.kind](state)


def tolerance(case):
    return "exact"


@functools.lru_cache(maxsize=None)
def _expected(fan, fail, record):
    """(children per parent, bytes per child that report a payload, share of all children's bytes that is assembled)"""
    r = np.random.default_rng(0)
    mu, sigma, lo, hi = FANS[fan]
    c = np.clip(np.rint(r.lognormal(mu, sigma, 200_000)), lo, hi)
    size = record or float(np.clip(np.rint(r.lognormal(7.5, 0.8, 200_000)), 256, 65536).mean())
    return float(c.mean()), size, float((c * (1 - fail) ** c).sum() / c.sum())


def work(case):
    """Bytes of the caller's arrays that a pass cannot do without: each input read once, each output written once."""
    kind = case["kind"]
    if kind == "nested":
        V, C = case["parents"], case["parents"] * 2.55
        F = C * 36
        n = 4 * V + 8 * V + 4 * C + 12 * C + 4 * (C + F) + 8 * F   # expansions and batches
        n += 18 * (C + F) + 17 * (V + C)                            # reports, verdicts, lists, outcomes, offsets
        return {"bytes": n + 4.0 * F * case["record"], "flops": 0.0}
    if kind == "stream":
        N, P = case["children"], case["children"] / math.exp(2.5 + 0.72)
        keep = _expected("stream", case["fail"], case["record"])[2]
        n = 13 * P + 8 * N + 4 * N + 4 * N + 18 * N + 17 * P
        return {"bytes": n + 2.0 * keep * N * case["record"], "flops": 0.0}
    if kind == "pass" and case["fan"] == "skew":
        heavy, size = _skew(case["parents"])
        P, N = case["parents"], case["parents"] - heavy + heavy * size
        S = N * case["record"] * 1.0
    else:
        fan, size, keep = _expected(case.get("fan", "docpage"), case.get("fail", 0.0), case.get("record") or 0)
        P, N = case["parents"], case["parents"] * fan
        S = keep * N * size
    expand = 12.0 * P + 8 * N
    if kind == "noalloc":
        return {"bytes": expand, "flops": 0.0}
    if kind == "bound":
        return {"bytes": expand + 8 * N, "flops": 0.0}
    if kind == "retry":
        return {"bytes": 8.0 * min(N, case["batch"] * case["batches"]), "flops": 0.0}
    lists = 17.0 * P
    if kind == "faults":
        return {"bytes": expand + 8 * N + 22 * N * (1 + 2 * case["repeats"]) + lists + 2 * S, "flops": 0.0}
    extra = 0.0
    if case.get("lists"):   # predicate and state; entries; half of the parents read again
        S *= 1 - case["drop"]
        extra = 3 * N + 13 * N + 8 * P + S + 6.5 * P
    return {"bytes": expand + 4 * N + 18 * N + lists + 2 * S + extra, "flops": 0.0}
