"""Kernels at the sizes where their splits can go wrong (edges of tiles and
groups, remainders, runs of parents without members), against the oracle;
every output compared exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


import paper_2609_18703_gb300 as ro  # noqa: E402
from tests.lockstep import Lockstep, dev, empty, host  # noqa: E402
from workload import DROPPED, FAILED, PRESENT  # noqa: E402


def _ones(n):
    return np.ones(n, np.uint32)


# counts, parents whose first child fails: the bitmap tiles hold 1,024 to 8,192
# parents (more than 4,096 completed in one are staged in groups), the plan's
# tiles 1,024 members, with up to 2,048 listed parents staged per tile
LISTS = {
    "one parent": (_ones(1), []),
    "plan tile - 1": (_ones(1023), []),
    "plan tile": (_ones(1024), []),
    "plan tile + 1": (_ones(1025), []),
    "word and tile remainders": (np.tile(np.array([1, 0, 3], np.uint32), 11_003), [0, 5, 33_008]),
    "groups of a full bitmap tile": (_ones(300_001), range(0, 300_001, 7)),
    "suppressed runs around one parent": (np.concatenate([_ones(5000), [1024], _ones(3000)]).astype(np.uint32),
                                          [*range(5000), *range(5001, 8001)]),
    "suppressed runs at plan tile edges": (np.concatenate([[1024], _ones(2500), [1024, 2048], _ones(9)])
                                           .astype(np.uint32), [*range(1, 2501), *range(2503, 2512)]),
    "every parent suppressed": (_ones(4097), range(4097)),
    "one parent over many tiles": (np.array([5000], np.uint32), []),
}


@pytest.mark.parametrize("name", LISTS)
@pytest.mark.parametrize("streams", [False, True])
def test_completed_list_and_plan(name, streams):
    counts, failing = LISTS[name]
    rng = np.random.default_rng(7)
    first = np.concatenate([[0], np.cumsum(counts.astype(np.int64))])
    n = int(first[-1])
    state = np.full(n, PRESENT, np.uint8)
    state[rng.random(n) < 0.1] = DROPPED
    fail = np.array([p for p in failing if counts[p]], np.int64)
    state[first[fail]] = FAILED
    length = rng.integers(0, 9, n).astype(np.uint32)
    off = np.concatenate([[0], np.cumsum(length[:-1])]).astype(np.uint64)
    arena = rng.integers(0, 256, int(length.sum()) + 16).astype(np.uint8)
    order = rng.permutation(n)
    with Lockstep(streams=streams) as ls:
        x = ls.expand(counts)["xid"]
        ls.batch_ready(x, 0, None, 64, flush=True)
        cursor = 0
        for part in np.array_split(order, 2):   # the second commit completes most parents
            ch = part.astype(np.uint32)
            cm = ls.commit(x, ch, state[ch], length[ch], off[ch], arena_bytes=arena.size)
            r = ls.assemble(x, arena, dev(arena, np.uint8), parents=None, n_parents=max(cm["n_done"], 1),
                            out_cap=cursor + arena.size, cursor=cursor)
            cursor += r["out_bytes"]
        ls.assemble(x, arena, dev(arena, np.uint8), parents=rng.permutation(counts.size)[:5000])
        ls.check_stats()


# a commit's fix-up spreads over the grid, 2,048 reports a CTA: repeated
# reports in every position (also of Grains an earlier commit sealed), wrong
# generations, GroupFailures that win or lose against a repeat, and reports
# after a barrier
@pytest.mark.parametrize("n", [33, 2047, 2048, 2049, 40_000])
@pytest.mark.parametrize("failures", [False, True])
@pytest.mark.parametrize("streams", [False, True])
def test_repeated_reports_over_many_ctas(n, failures, streams):
    rng = np.random.default_rng(n)
    counts = rng.integers(1, 40, max(2, n // 12)).astype(np.uint32)
    N = int(counts.sum())
    with Lockstep(streams=streams) as ls:
        x = ls.expand(counts)["xid"]
        ls.batch_ready(x, 0, rng.permutation(N)[: N - N // 10], 16)   # some stay queued, some are never named
        for _ in range(3):
            ch = rng.integers(0, N // 2 + 1 if n > 2048 else N, n).astype(np.uint32)
            st = rng.choice([PRESENT, PRESENT, PRESENT, DROPPED, FAILED, 0], n).astype(np.uint8)
            if failures:
                st[rng.random(n) < 0.003] = 5
            gen = (rng.random(n) < 0.1).astype(np.uint32)
            ls.commit(x, ch, st, rng.integers(0, 100, n).astype(np.uint32), rng.integers(0, 1 << 20, n).astype(np.uint64),
                      gen=gen, arena_bytes=1 << 21)
            ls.batch_ready(x, 0, rng.permutation(N)[: N // 3], 16)
        ls.check_stats()


# the queue window: recovery groups ahead of queued entries, slices of 2,048 a
# CTA, sealed entries in either, what stays queued and what is refused
@pytest.mark.parametrize("n", [1, 31, 2047, 2048, 2049, 9000])
@pytest.mark.parametrize("sealed", [False, True])
def test_window_over_many_ctas(n, sealed):
    rng = np.random.default_rng(n)
    counts = rng.integers(1, 9, 6000).astype(np.uint32)
    N = int(counts.sum())
    off = np.concatenate([[0], np.cumsum(counts)])
    order = rng.permutation(N)
    with Lockstep() as ls:
        x = ls.expand(counts)["xid"]
        ls.batch_ready(x, 0, order[: N // 2], 7, flush=True)
        ls.batch_ready(x, 0, order[N // 2: N // 2 + 5], 1000)   # five stay queued
        retried = order[: min(n, N // 2)]
        ls.retry(x, 0, retried)
        if sealed:   # the parents of some in-flight Grains fail: their retried and queued siblings are sealed
            ch = order[N // 2 - 40: N // 2].astype(np.uint32)
            ls.commit(x, ch, np.full(ch.size, 5, np.uint8), np.zeros(ch.size, np.uint32), np.zeros(ch.size, np.uint64))
            ls.commit(x, order[N // 2:N // 2 + 3].astype(np.uint32), np.full(3, 5, np.uint8), np.zeros(3, np.uint32),
                      np.zeros(3, np.uint64))
        more = np.concatenate([order[N // 2 + 5: N // 2 + 300], order[N // 2 + 5: N // 2 + 20]])
        ls.batch_ready(x, 0, more[:0], 1, cap=0, flush=True)          # refused: the window stays
        ls.batch_ready(x, 0, more[:100], max(1, n // 2 + 3), cap=N)   # part of the recovery group, maybe, stays
        ls.retry(x, 0, order[N // 4: N // 4 + 50])
        ls.batch_ready(x, 0, more, n + 400, cap=N)
        ls.batch_ready(x, 0, None, 64, flush=True)
        ls.check_stats()
        assert off[-1] == N


# the expansion's scan: tiles of 1,024 parents up to 131,072 of them, of 4,096
# beyond; fill tiles of 4,096 children
@pytest.mark.parametrize("P", [1, 1023, 1024, 1025, 4097, 131_072, 131_073, 135_167, 300_001])
@pytest.mark.parametrize("kind", ["ones", "sparse", "mixed", "heavy"])
def test_expansion_tiles(P, kind):
    rng = np.random.default_rng(P)
    if kind == "ones":
        counts = _ones(P)
    elif kind == "sparse":
        counts = (rng.random(P) < 0.02).astype(np.uint32)
    else:
        counts = rng.integers(0, 6, P).astype(np.uint32)
        if kind == "heavy":
            counts[rng.integers(0, P, 3)] = rng.integers(4000, 20_000, 3)
    n = int(counts.sum())
    with Lockstep() as ls:
        r = ls.expand(counts)   # compares offsets, parents, ordinals and empties
        d_off, d_p, d_o = empty(P + 1, np.uint64), empty(n, np.uint32), empty(n, np.uint32)
        d_e = empty(P, np.uint32)
        # (the caller's arrays at their least alignment)
        d_c = dev(np.concatenate([[7], counts]), np.uint32)[1:]
        st, k, e = ro.ro_expand_noalloc(d_c, P, d_off, d_p, d_o, n, d_e)
        assert (st, k, e) == (ro.RO_OK, n, r["n_empty"])
        off = r["offsets"].astype(np.int64)
        assert np.array_equal(host(d_off, np.uint64, P + 1), r["offsets"])
        assert np.array_equal(host(d_p, np.uint32, n), np.repeat(np.arange(P), counts))
        assert np.array_equal(host(d_o, np.uint32, n), np.arange(n) - np.repeat(off[:-1], counts))
        assert np.array_equal(host(d_e, np.uint32, e), np.flatnonzero(counts == 0))


# the copy of small records: words inside one member, over member boundaries,
# over many one-byte members; ranges cut at slices (direct) and chunks
@pytest.mark.parametrize("lo,hi", [(1, 1), (1, 5), (15, 17), (16, 16), (17, 17), (32, 32), (48, 48), (0, 200), (128, 128)])
@pytest.mark.parametrize("chunks", [True, False])
def test_copy_of_small_records(lo, hi, chunks, monkeypatch):
    monkeypatch.setenv("RO_COPY_SMALL_CHUNKS", "0" if chunks else "256")
    rng = np.random.default_rng(lo * 1000 + hi)
    counts = rng.integers(0, 60, 1500).astype(np.uint32)
    counts[700] = 3001
    n = int(counts.sum())
    state = np.full(n, PRESENT, np.uint8)
    state[rng.random(n) < 0.05] = DROPPED
    state[rng.random(n) < 0.001] = FAILED
    length = rng.integers(lo, hi + 1, n).astype(np.uint32)
    if lo != hi:
        length[rng.integers(0, n, 2)] = 30_000   # members larger than a unit among them
    order = rng.permutation(n)
    off = np.zeros(n, np.uint64)
    off[order] = np.concatenate([[0], np.cumsum(length[order][:-1])])
    arena = rng.integers(0, 256, int(length.sum())).astype(np.uint8)
    for cursor in (0, 5):
        with Lockstep() as ls:
            x = ls.expand(counts)["xid"]
            ls.batch_ready(x, 0, None, 64, flush=True)
            cm = ls.commit(x, order.astype(np.uint32), state[order], length[order], off[order], arena_bytes=arena.size)
            ls.assemble(x, arena, dev(arena, np.uint8), parents=None, n_parents=cm["n_done"],
                        out_cap=cursor + arena.size, cursor=cursor)
            ls.assemble(x, arena, dev(arena, np.uint8), parents=rng.permutation(counts.size)[:900])


# chunks of more pieces than a stage's table holds, in a call whose records
# average too large to be gathered
@pytest.mark.parametrize("cursor", [0, 11])
def test_copy_of_clustered_small_records(cursor):
    rng = np.random.default_rng(cursor)
    counts = np.where(np.arange(440) % 11 == 0, 3000, 20).astype(np.uint32)
    n = int(counts.sum())
    tiny = np.repeat(counts == 3000, counts)
    length = np.where(tiny, rng.integers(4, 13, n), rng.integers(2900, 3100, n)).astype(np.uint32)
    order = rng.permutation(n)
    off = np.zeros(n, np.uint64)
    off[order] = np.concatenate([[0], np.cumsum(length[order][:-1], dtype=np.uint64)])
    arena = rng.integers(0, 256, int(length.sum(dtype=np.uint64))).astype(np.uint8)
    with Lockstep() as ls:
        x = ls.expand(counts)["xid"]
        ls.batch_ready(x, 0, None, 64, flush=True)
        cm = ls.commit(x, order.astype(np.uint32), np.full(n, PRESENT, np.uint8), length[order], off[order],
                       arena_bytes=arena.size)
        ls.assemble(x, arena, dev(arena, np.uint8), parents=None, n_parents=cm["n_done"],
                    out_cap=cursor + arena.size, cursor=cursor)


# chunks of more members than a producer fetches ahead (65), of records too
# large to be gathered: the staged copy's piece table over several rounds
@pytest.mark.parametrize("lo,hi", [(141, 160), (60, 400), (250, 260)])
@pytest.mark.parametrize("pinned", [False, True])
def test_copy_of_chunks_with_many_pieces(lo, hi, pinned, monkeypatch):
    monkeypatch.setenv("RO_COPY_SMALL_CHUNKS", "0")
    rng = np.random.default_rng(lo)
    counts = rng.integers(0, 60, 1500).astype(np.uint32)
    n = int(counts.sum())
    state = np.full(n, PRESENT, np.uint8)
    state[rng.random(n) < 0.03] = DROPPED
    length = rng.integers(lo, hi + 1, n).astype(np.uint32)
    order = rng.permutation(n)
    off = np.zeros(n, np.uint64)
    off[order] = np.concatenate([[0], np.cumsum(length[order][:-1])])
    arena = rng.integers(0, 256, int(length.sum())).astype(np.uint8)
    d_arena = torch.from_numpy(arena).pin_memory() if pinned else dev(arena, np.uint8)
    for cursor in (0, 9):
        with Lockstep() as ls:
            x = ls.expand(counts)["xid"]
            ls.batch_ready(x, 0, None, 64, flush=True)
            cm = ls.commit(x, order.astype(np.uint32), state[order], length[order], off[order], arena_bytes=arena.size)
            ls.assemble(x, arena, d_arena, parents=None, n_parents=cm["n_done"], out_cap=cursor + arena.size, cursor=cursor)


# parents: sort digits of up to 10 bits (no pass, 1, 2, 3 of them, and the
# first id of one more); queued: edges of the sort's 2,048-entry tiles and the
# reservation scan's 4,096
@pytest.mark.parametrize("P", [1, 2, 1024, 1025, (1 << 20) + 1])
@pytest.mark.parametrize("n", [1, 2047, 2049, 4096, 4097, 20_000])
@pytest.mark.parametrize("sealed", [False, True])
def test_parent_bound_windows(P, n, sealed):
    rng = np.random.default_rng(n + P)
    counts = np.zeros(P, np.uint32)
    counts[[0, -1]] = n // 2 + 1   # the smallest and the largest parent id
    counts[rng.integers(0, P, n)] += 1
    N = int(counts.sum())
    order = rng.permutation(N).astype(np.uint32)
    with Lockstep() as ls:
        x = ls.expand(counts)["xid"]
        ls.batch_ready_parent(x, 0, order[:n], N + 1)   # nothing leaves: n entries stay queued
        if sealed:   # the first one's parent fails: its queued siblings leave the queue
            ls.commit(x, order[:1], np.full(1, 5, np.uint8), np.zeros(1, np.uint32), np.zeros(1, np.uint64))
        ls.batch_ready_parent(x, 0, order[n:n + 7], 3)   # the window, up to the first short batch
        ls.batch_ready_parent(x, 0, None, 3, flush=True)
        ls.check_stats()


# copies one behind another without a wait, each starting at the cursor the one
# before it left, with refused ones between (which leave it alone)
@pytest.mark.parametrize("lo,hi", [(1, 60), (400, 700)])   # gathered; copied a member at a time
@pytest.mark.parametrize("streams", [False, True])
def test_copies_in_a_row(lo, hi, streams):
    rng = np.random.default_rng(lo)
    W, n = 80, 40   # waves, parents of one child each completed by a wave
    N = W * n
    length = rng.integers(lo, hi + 1, N).astype(np.uint32)
    off = np.concatenate([[0], np.cumsum(length[:-1])]).astype(np.uint64)
    arena = rng.integers(0, 256, int(length.sum())).astype(np.uint8)
    order = rng.permutation(N).astype(np.uint32)
    want = []
    with Lockstep(streams=streams) as ls:
        x = ls.expand(_ones(N))["xid"]
        ls.batch_ready(x, 0, None, 64, flush=True)
        d_arena, d_child = dev(arena, np.uint8), dev(order, np.uint32)
        d_state, d_len, d_off = dev(np.full(N, PRESENT), np.uint8), dev(length[order], np.uint32), dev(off[order], np.uint64)
        d_status, d_oo = empty(W * n, np.uint8), empty(W * (n + 1), np.uint64)
        out, cursor = empty(arena.size, np.uint8), empty(1, np.uint64)
        torch.cuda.synchronize()
        refused = rng.random(W) < 0.3
        for w in range(W):
            at = lambda t, i, size: t.data_ptr() + i * size   # noqa: E731
            st, _ = ro.ro_gather_commit(ls.ctx, x, n, None, at(d_child, w * n, 4), at(d_state, w * n, 1),
                                        at(d_len, w * n, 4), at(d_off, w * n, 8), None, arena.size, want_host=False)
            assert st == ro.RO_OK
            st, _ = ro.ro_assemble(ls.ctx, x, d_arena, arena.size, None, n, None, at(d_status, w * n, 1),
                                   at(d_oo, w * (n + 1), 8), None, out, 0 if refused[w] else arena.size, cursor,
                                   want_host=False)
            assert st == ro.RO_OK
            if not refused[w]:
                done = np.sort(order[w * n:(w + 1) * n])
                want += [arena[int(off[c]):int(off[c]) + int(length[c])] for c in done]
        assert ro.ro_ctx_sync(ls.ctx) == (ro.RO_E_CAPACITY if refused.any() else ro.RO_OK)
        want = np.concatenate(want)
        assert int(host(cursor, np.uint64, 1)[0]) == want.size
        assert np.array_equal(host(out, np.uint8, want.size), want)


# several Calls' queue windows in one launch, each over many CTAs: one Call's
# recovery group beside others' few entries, sealed entries in one of them (it
# compacts while the others' leave in place), repeats, a refused Call, and the
# windows that these leave for the next calls
@pytest.mark.parametrize("n_calls", [2, 4])
@pytest.mark.parametrize("n", [2049, 6000])
@pytest.mark.parametrize("sealed", [False, True])
def test_windows_of_several_calls_over_many_ctas(n_calls, n, sealed):
    rng = np.random.default_rng(n + n_calls)
    counts = rng.integers(1, 9, 24_000).astype(np.uint32)
    N = int(counts.sum())
    calls_of = (np.arange(counts.size) % n_calls).astype(np.uint8)
    order = rng.permutation(N).astype(np.uint32)
    call = np.repeat(calls_of, counts)[order]
    every, last, half = list(range(n_calls)), n_calls - 1, N // 2
    mine = [order[:half][call[:half] == c] for c in every]   # dispatched first
    assert mine[0].size > 2 * n and mine[last].size > 2 * n
    with Lockstep(n_calls=n_calls) as ls:
        x = ls.expand(counts, parent_call=calls_of)["xid"]
        ls.batch_ready_calls(x, every, order[:half], 7, flush=True)
        ls.batch_ready_calls(x, every, order[half:half + 40], 1000)   # a few stay queued
        ls.retry(x, 0, mine[0][:n])
        if sealed:   # parents of some dispatched and some queued Grains fail
            ch = np.concatenate([mine[0][-40:], mine[last][-3:]])
            ls.commit(x, ch, np.full(ch.size, 5, np.uint8), np.zeros(ch.size, np.uint32), np.zeros(ch.size, np.uint64))
        more = np.concatenate([order[half + 40:half + 900], order[half + 40:half + 60], [N + 3]]).astype(np.uint32)
        ls.batch_ready_calls(x, every, more, 64, caps=[10] + [N] * last)   # Call 0 is refused, its group stays
        ls.retry(x, last, mine[last][n // 2:n // 2 + n])
        ls.batch_ready_calls(x, every[::-1], more[:0], 100)   # windows alone, what is over stays
        ls.retry(x, 0, mine[0][n:n + n])
        ls.batch_ready_calls(x, every, order[half:], 3000)
        ls.batch_ready_calls(x, every, order[half:half + 5000], 6000, caps=[N] * last + [0])
        ls.retry(x, last, mine[last][:n])
        ls.batch_ready_calls(x, every, None, 64, flush=True)
        ls.check_stats()


# the commit's fix-up behind the scatter of a context of several Calls (its
# fence and its publish are separate transactions)
@pytest.mark.parametrize("n", [2049, 40_000])
@pytest.mark.parametrize("failures", [False, True])
def test_repeated_reports_of_several_calls(n, failures):
    rng = np.random.default_rng(n + 1)
    counts = rng.integers(1, 40, n // 12).astype(np.uint32)
    N = int(counts.sum())
    with Lockstep(n_calls=3, streams=True) as ls:
        x = ls.expand(counts, parent_call=(np.arange(counts.size) % 3).astype(np.uint8))["xid"]
        ls.batch_ready_calls(x, [0, 1, 2], rng.permutation(N)[: N - N // 10], 16)
        for _ in range(3):
            ch = rng.integers(0, N // 2 + 1 if n > 2049 else N, n).astype(np.uint32)
            st = rng.choice([PRESENT, PRESENT, PRESENT, DROPPED, FAILED, 0], n).astype(np.uint8)
            if failures:
                st[rng.random(n) < 0.003] = 5
            gen = (rng.random(n) < 0.1).astype(np.uint32)
            ls.commit(x, ch, st, rng.integers(0, 100, n).astype(np.uint32), rng.integers(0, 1 << 20, n).astype(np.uint64),
                      gen=gen, arena_bytes=1 << 21)
            ls.batch_ready_calls(x, [2, 0, 1], rng.permutation(N)[: N // 3], 16)
        ls.check_stats()


# an output of exactly the assembled bytes, and lists that an arena too small
# makes void, while another stream's kernels keep copies' CTAs waiting for room
def test_tight_output_beside_other_work():
    rng = np.random.default_rng(3)
    W, n = 60, 50
    N = W * n
    length = rng.integers(300, 900, N).astype(np.uint32)
    off = np.concatenate([[0], np.cumsum(length[:-1])]).astype(np.uint64)
    arena = rng.integers(0, 256, int(length.sum())).astype(np.uint8)
    order = rng.permutation(N).astype(np.uint32)
    want = np.concatenate([arena[int(off[c]):int(off[c]) + int(length[c])]
                           for w in range(W) for c in np.sort(order[w * n:(w + 1) * n])])
    with Lockstep(streams=True) as ls:
        d_arena, d_child, d_counts = dev(arena, np.uint8), dev(order, np.uint32), dev(_ones(N), np.uint32)
        d_state, d_len, d_off = dev(np.full(N, PRESENT), np.uint8), dev(length[order], np.uint32), dev(off[order], np.uint64)
        d_all = dev(np.arange(N), np.uint32)
        eo, ep, eord, eb = empty(N + 1, np.uint64), empty(N, np.uint32), empty(N, np.uint32), empty(N, np.uint32)
        d_status, d_oo, out, cursor = empty(N, np.uint8), empty(N + W, np.uint64), empty(arena.size, np.uint8), empty(1, np.uint64)
        x_status, x_oo, x_out = empty(N, np.uint8), empty(N + 1, np.uint64), empty(arena.size, np.uint8)
        busy, load = torch.cuda.Stream(), torch.zeros(1 << 27, device="cuda")
        torch.cuda.synchronize()
        for again in range(8):
            with torch.cuda.stream(busy):
                for _ in range(40):
                    load.add_(1.0)
            assert ro.ro_ctx_reset(ls.ctx) == ro.RO_OK
            cursor.zero_()
            st, k, _, x = ro.ro_expand(ls.ctx, -1, d_counts, N, None, eo, ep, eord, N)
            assert st == ro.RO_OK and k == N
            assert ro.ro_batch_ready(ls.ctx, x, 0, None, 0, 64, True, eb, N, None, want_host=False)[0] == ro.RO_OK
            for w in range(W):
                at = lambda t, i, size: t.data_ptr() + i * size   # noqa: E731
                st, _ = ro.ro_gather_commit(ls.ctx, x, n, None, at(d_child, w * n, 4), at(d_state, w * n, 1),
                                            at(d_len, w * n, 4), at(d_off, w * n, 8), None, arena.size, want_host=False)
                assert st == ro.RO_OK
                st, _ = ro.ro_assemble(ls.ctx, x, d_arena, arena.size, None, n, None, at(d_status, w * n, 1),
                                       at(d_oo, w * (n + 1), 8), None, out, arena.size, cursor, want_host=False)
                assert st == ro.RO_OK
            assert ro.ro_ctx_sync(ls.ctx) == ro.RO_OK, ro.ro_last_error(ls.ctx)
            assert int(host(cursor, np.uint64, 1)[0]) == arena.size
            assert np.array_equal(host(out, np.uint8, arena.size), want)
            for size, status in ((arena.size // 2, ro.RO_E_INVAL), (arena.size, ro.RO_OK)):
                for _ in range(3):
                    assert ro.ro_assemble(ls.ctx, x, d_arena, size, d_all, N, None, x_status, x_oo, None, x_out,
                                          arena.size, None, None, want_host=False)[0] == ro.RO_OK
                assert ro.ro_ctx_sync(ls.ctx) == status, ro.ro_last_error(ls.ctx)
            assert np.array_equal(host(x_out, np.uint8, arena.size), arena)
            x_out.zero_()
            out.zero_()
