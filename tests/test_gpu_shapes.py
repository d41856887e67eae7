"""The kernels' dispatch at the sizes where it can go wrong: edges of tiles, remainders, the smallest and largest of a
range, and the branches between kernels, each against the fp64 checker."""
import dataclasses

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _wl(config, **kw):
    from paper_2510_09608_b200 import streamgen as sg
    return dataclasses.replace(sg.workloads()[config], **kw)


# --- chunk prefill: units cut between thread blocks (caches of 18 pages and more), one head per KV head (no shared
# --- rotation factors), ragged row tiles, a chunk longer than the windows keep, positions beyond 2^16
@pytest.mark.parametrize("d,hq,hk,frames,vw,base,contiguous", [
    (128, 28, 4, 1, 2304, 0, True), (128, 4, 4, 3, 1984, 0, True), (64, 7, 1, 3, 2304, 0, True), (64, 16, 8, 1, 2000, 0, True),
    (128, 28, 4, 9, 192, 0, True), (64, 12, 2, 7, 64, 0, True), (128, 6, 2, 2, 512, 70000, False)])
def test_chunk_prefill_work_split(d, hq, hk, frames, vw, base, contiguous):
    from harness import SideBySide, assert_close
    wl = _wl(2, layers=1, q_heads=hq, kv_heads=hk, head_dim=d, sections=(d // 8, d // 16 * 3, d // 16 * 3), n_sink=40, vision_window=vw, text_window=70,
             frames=frames, grid_h=8, grid_w=9, text_max=21)
    s = SideBySide(wl, contiguous=contiguous)
    s.stream.base = base
    for _ in range(2 + (vw + 70) // (72 * frames)):
        s.append_chunk()
        s.evict()
    s.append_chunk()
    s.evict()
    s.check_metadata()
    n = len(s.last[0])
    rows = sorted({0, 1, n // 2, n - 2, n - 1, *range(0, n, 37)})
    assert_close(s.attend(0, rows=rows))


# --- page lists longer than what a thread block keeps of one (96 entries), and the pages of other caches than its first one's:
# --- chunks of several units per thread block in one launch over caches of different lengths
@pytest.mark.parametrize("d,hq,hk", [(64, 7, 1), (128, 6, 2)])
def test_chunk_prefill_of_many_pages(d, hq, hk):
    from harness import SideBySide, assert_close
    wl = _wl(2, layers=1, q_heads=hq, kv_heads=hk, head_dim=d, sections=(d // 8, d // 16 * 3, d // 16 * 3), n_sink=40, vision_window=13000, text_window=70,
             frames=15, grid_h=8, grid_w=9, text_max=21)
    s = SideBySide(wl)
    for _ in range(13):
        s.append_chunk()
        s.evict()
    assert_close(s.attend(0, rows=list(range(0, len(s.last[0]), 61))))


def test_chunk_prefill_of_several_caches_at_once():
    from paper_2510_09608_b200 import binding
    gen = torch.Generator(device="cuda").manual_seed(11)
    normal = lambda *shape: torch.randn(*shape, generator=gen, device="cuda", dtype=torch.bfloat16)      # noqa: E731
    hq, hk, d = 28, 4, 128
    caches, q, pos, want, n_q = [], [], [], [], [1500, 37, 2100, 900]
    for n, kept in zip(n_q, (3000, 14000, 2500, 6000)):
        c = binding.Cache(1, hk, d, 64, 14000, 100, 14300)
        c.append(0, normal(kept, hk, d), normal(kept, hk, d), torch.ones(kept, dtype=torch.uint8, device="cuda"), torch.arange(kept, dtype=torch.int32, device="cuda"))
        caches.append(c)
        q.append(normal(n, hq, d))
        pos.append(torch.arange(kept - n, kept, dtype=torch.int32, device="cuda"))
        want.append(c.attend(0, q[-1], pos[-1]).clone())
    out = torch.empty(sum(n_q), hq, d, dtype=torch.bfloat16, device="cuda")
    binding.attend_batched_varlen(caches, 0, torch.cat(q), torch.cat(pos), n_q, out)
    at = 0
    for n, w in zip(n_q, want):
        # the cuts lie elsewhere, so weights are rounded to bf16 against other reference maxima: 2^-9 of a weight each, and outputs (below 1 in
        # size here) to bf16 once more
        assert (out[at:at + n].float() - w.float()).abs().max() < 2e-2
        at += n
    assert all(c.status() == binding.OK for c in caches)


def test_chunk_prefill_of_several_caches_against_the_checker():
    """Rows of every cache against the checker.  A page of 128 left out or counted twice moves the outputs over 14,000 keys by a tenth of
    their rms size, no causal limit moves the first rows by a twentieth and more: outside the 2 % that are allowed."""
    import oracle
    from harness import SideBySide, assert_close, bits_to_dev, dev_to_f64
    from paper_2510_09608_b200 import binding
    gen = torch.Generator().manual_seed(11)
    bits = lambda *shape: torch.randn(*shape, generator=gen).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)      # noqa: E731
    hq, hk, d = 28, 4, 128
    caches, refs, q, pos, n_q = [], [], [], [], [1500, 37, 2100, 900]
    for n, kept in zip(n_q, (3000, 14000, 2500, 6000)):
        c, ref = binding.Cache(1, hk, d, 64, 14000, 100, 14300), oracle.Oracle(1, hk, d, 64, 14000, 100)
        c.set_rope(binding.ROPE_1D, 1.0e4)
        k, v, types, ps = bits(kept, hk, d), bits(kept, hk, d), np.ones(kept, np.uint8), np.arange(kept, dtype=np.int32)
        c.append(0, bits_to_dev(k), bits_to_dev(v), torch.from_numpy(types).cuda(), torch.from_numpy(ps).cuda())
        ref.append(k[None], v[None], types, ps)
        caches.append(c)
        refs.append(ref)
        q.append(bits(n, hq, d))
        pos.append(ps[-n:])
    out = torch.empty(sum(n_q), hq, d, dtype=torch.bfloat16, device="cuda")
    binding.attend_batched_varlen(caches, 0, bits_to_dev(np.concatenate(q)), torch.from_numpy(np.concatenate(pos)).cuda(), n_q, out)
    at = 0
    for c, ref, n, x, ps in zip(caches, refs, n_q, q, pos):
        assert c.status() == binding.OK
        rows = sorted({0, 1, 36, n // 2, n - 1, *range(5, n, 211)})
        # row by row: another row's error does not hide one's own
        got, want = dev_to_f64(out[at:at + n])[rows], ref.attend(0, x, ps, rows)
        for r in range(len(rows)):
            assert_close(SideBySide._stats(got[r], want[r]))
        at += n


# --- chunks of few rows: rows at the edges of a 16-row tile, one to eight thread blocks over the keys, two tiles per block,
# --- partly filled pages, positions beyond 2^16
@pytest.mark.parametrize("d,hq,hk,frames,gh,gw,vw,base,contiguous", [
    (64, 4, 1, 1, 2, 2, 64, 0, True), (128, 4, 4, 1, 1, 15, 70, 0, True), (128, 4, 4, 1, 1, 17, 330, 0, True), (64, 1, 1, 1, 1, 2, 30, 0, True),
    (64, 4, 1, 1, 6, 6, 2300, 0, True), (128, 8, 4, 1, 6, 6, 2300, 0, True), (64, 16, 8, 1, 6, 6, 2300, 0, True), (128, 28, 4, 1, 5, 6, 2000, 0, True),
    (64, 16, 8, 2, 8, 10, 500, 0, True), (128, 28, 4, 2, 8, 8, 300, 0, True), (128, 9, 1, 1, 3, 5, 200, 70000, False), (64, 3, 1, 1, 5, 5, 20, 0, True)])
def test_chunk_prefill_of_few_rows(d, hq, hk, frames, gh, gw, vw, base, contiguous):
    from harness import SideBySide, assert_close
    wl = _wl(2, layers=1, q_heads=hq, kv_heads=hk, head_dim=d, sections=(d // 8, d // 16 * 3, d // 16 * 3), n_sink=5, vision_window=vw, text_window=37,
             frames=frames, grid_h=gh, grid_w=gw, text_max=2)
    s = SideBySide(wl, contiguous=contiguous)
    s.stream.base = base
    for _ in range(2 + vw // (frames * gh * gw)):
        s.append_chunk()
        s.evict()
    for _ in range(2):
        s.append_chunk()
        s.evict()
        assert_close(s.attend(0))


# --- the tensor-core prefill kernel's waits made to run out (the few rows of other give-up tests are the small kernel's)
@pytest.mark.parametrize("d,hq,hk", [(128, 28, 4), (64, 12, 2)])
def test_large_chunk_prefill_gives_up_and_recovers(d, hq, hk):
    from harness import SideBySide, assert_close, bits_to_dev, dev_to_f64
    from paper_2510_09608_b200 import binding
    wl = _wl(2, layers=1, q_heads=hq, kv_heads=hk, head_dim=d, sections=(d // 8, d // 16 * 3, d // 16 * 3), n_sink=40, vision_window=2304, text_window=70,
             frames=9, grid_h=8, grid_w=9, text_max=21)
    s = SideBySide(wl)
    for _ in range(5):
        s.append_chunk()
        s.evict()
    gids, _, pos = s.last
    Q, qp = bits_to_dev(s.stream.q(0, gids)), torch.from_numpy(np.ascontiguousarray(pos)).cuda()
    s.cache.debug_set_wait_limit(0)
    s.cache.attend(0, Q, qp)
    assert s.cache.status() == binding.ERR_TIMEOUT
    s.cache.debug_set_wait_limit(1 << 20)
    out = dev_to_f64(s.cache.attend(0, Q, qp))
    s._give_values_to_ref(0)
    rows = list(range(0, len(gids), 29))
    assert_close(s._stats(out[rows], s.ref.attend(0, s.stream.q(0, gids), pos, rows=rows)))


# --- waits that run out somewhere in the middle of a unit: some polls, but too few for most waits.  The thread blocks come to their
# --- end whoever gave up first, and the caches serve again
@pytest.mark.parametrize("d,hq,hk", [(128, 28, 4), (64, 12, 2)])
def test_large_chunk_prefill_gives_up_in_the_middle(d, hq, hk):
    from paper_2510_09608_b200 import binding
    gen = torch.Generator(device="cuda").manual_seed(7)
    normal = lambda *shape: torch.randn(*shape, generator=gen, device="cuda", dtype=torch.bfloat16)      # noqa: E731
    kept, n_q = 3000, 1400                                 # (several units per thread block)
    c = binding.Cache(1, hk, d, 64, kept, 100, kept + 300)
    c.append(0, normal(kept, hk, d), normal(kept, hk, d), torch.ones(kept, dtype=torch.uint8, device="cuda"), torch.arange(kept, dtype=torch.int32, device="cuda"))
    q, pos = normal(n_q, hq, d), torch.arange(kept - n_q, kept, dtype=torch.int32, device="cuda")
    want = c.attend(0, q, pos).clone()
    seen = 0
    for limit in (1, 2, 3, 5, 8, 13, 21, 34, 70):
        c.debug_set_wait_limit(limit)
        c.attend(0, q, pos)
        status = c.status()
        assert status in (binding.OK, binding.ERR_TIMEOUT)
        seen += status == binding.ERR_TIMEOUT
        c.debug_set_wait_limit(1 << 20)
        assert torch.equal(c.attend(0, q, pos), want)
    assert seen


# --- pieces of a cut unit that do not wait for one another: the poll limit leaves the other waits alone and the meeting none,
# --- so that whoever comes last puts the others' shares together; the same bits as when each merges its own
@pytest.mark.parametrize("d,hq,hk,frames,vw", [(128, 28, 4, 7, 2304), (128, 28, 4, 1, 6000), (64, 12, 2, 7, 2304), (64, 16, 8, 1, 9000)])
def test_cut_units_without_waiting(d, hq, hk, frames, vw):
    from harness import SideBySide, bits_to_dev
    from paper_2510_09608_b200 import binding
    wl = _wl(2, layers=1, q_heads=hq, kv_heads=hk, head_dim=d, sections=(d // 8, d // 16 * 3, d // 16 * 3), n_sink=40, vision_window=vw, text_window=70,
             frames=frames, grid_h=8, grid_w=9, text_max=21)
    s = SideBySide(wl)
    for _ in range(2 + (vw + 70) // (72 * frames)):
        s.append_chunk()
        s.evict()
    gids, _, pos = s.last
    Q, qp = bits_to_dev(s.stream.q(0, gids)), torch.from_numpy(np.ascontiguousarray(pos)).cuda()
    s._give_values_to_ref(0)
    rows = list(range(0, len(gids), 31))
    want = s.ref.attend(0, s.stream.q(0, gids), pos, rows=rows)
    out = s.cache.attend(0, Q, qp).clone()
    s.cache.debug_set_wait_limit((1 << 14) - 1)
    for _ in range(3):                                     # (the counters come back to zero)
        again = s.cache.attend(0, Q, qp)
        assert torch.equal(out, again)
    s.cache.debug_set_wait_limit(1 << 20)
    assert torch.equal(out, s.cache.attend(0, Q, qp)) and s.cache.status() == binding.OK
    from harness import assert_close, dev_to_f64
    assert_close(s._stats(dev_to_f64(out)[rows], want))


def test_cut_units_of_two_streams_at_once():
    """Two caches on two streams: pieces of one launch wait for others whose thread blocks the other launch keeps from running.
    The same bits as one after the other."""
    from paper_2510_09608_b200 import binding
    gen = torch.Generator(device="cuda").manual_seed(4)
    normal = lambda *shape: torch.randn(*shape, generator=gen, device="cuda", dtype=torch.bfloat16)      # noqa: E731
    made = []
    for hq, hk, n_q, kept in ((16, 2, 390, 8000), (28, 4, 133, 4500)):
        c = binding.Cache(2, hk, 128, 64, kept, 100, kept + 300)
        c.append(-1, normal(2, kept, hk, 128), normal(2, kept, hk, 128), torch.ones(kept, dtype=torch.uint8, device="cuda"),
                 torch.arange(kept, dtype=torch.int32, device="cuda"))
        q, pos = normal(2, n_q, hq, 128), torch.arange(kept - n_q, kept, dtype=torch.int32, device="cuda")
        want = [c.attend(l, q[l], pos) for l in range(2)]
        torch.cuda.synchronize()
        c.set_stream(torch.cuda.Stream())
        made.append((c, q, pos, want, [torch.empty_like(q) for _ in range(6)]))
    torch.cuda.synchronize()
    for rep in range(6):
        for l in range(2):
            for c, q, pos, _, outs in made:
                c.attend(l, q[l], pos, outs[rep][l])
    torch.cuda.synchronize()
    for c, _, _, want, outs in made:
        assert c.status() == binding.OK
        assert all(torch.equal(out[l], want[l]) for out in outs for l in range(2))


# --- append metadata: one token, up to 1024 (one per thread), more; sinks of either rule that end inside a chunk; evictions
# --- of more tokens than fit the lists in shared memory
@pytest.mark.parametrize("sink_any", [False, True])
@pytest.mark.parametrize("sizes", [(1, 31, 32, 33, 96, 97, 128), (1023, 1024, 1025, 2), (1500, 900, 1, 1700, 40)])
def test_append_sizes_and_large_evictions(sizes, sink_any):
    from harness import SideBySide
    wl = _wl(2, layers=1, q_heads=2, kv_heads=1, head_dim=64, rope_mode=0, sections=(32, 0, 0), n_sink=60, vision_window=150, text_window=130)
    s = SideBySide(wl, capacity=6000, sink_any=sink_any)
    rng = np.random.default_rng(sum(sizes))
    gid = pos = 0
    for rep in range(2):
        for i, n in enumerate(sizes):
            types = rng.integers(0, 2, n).astype(np.uint8)
            s._append(np.arange(gid, gid + n), types, (pos + np.arange(n)).astype(np.int32))
            gid, pos = gid + n, pos + n
            s.check_metadata()
            if i % 3 == 2 or i == len(sizes) - 1:
                s.evict()
                s.check_metadata()
    s.check_kv(0)


# --- appends and evictions of small caches in one launch each, at the lines to the two-launch forms: as many new rows as one
# --- block writes and one more, as many kept tokens as it re-rotates and one more, all layers at once, positions beyond 2^16
@pytest.mark.parametrize("over", [0, 1])
@pytest.mark.parametrize("d,hk,layers,sizes,capacity,base,contiguous", [
    (64, 1, 1, (37, 64, 65, 1, 31), 256, 0, True), (128, 2, 1, (16, 17, 1, 3), 200, 0, True), (64, 1, 3, (21, 22, 33, 2), 100, 0, True),
    (64, 2, 2, (1, 2, 16, 17), 100, 70000, False), (128, 1, 2, (7, 15, 16, 17), 70, 70000, True), (64, 1, 1, (40, 300), 2600, 0, True)])
def test_small_caches_in_one_launch(d, hk, layers, sizes, capacity, base, contiguous, over):
    from harness import SideBySide
    keep = 16384 // (d * hk * layers) + over                  # tokens the windows keep: one block re-rotates them, or a launch of its own
    wl = _wl(2, layers=layers, q_heads=hk, kv_heads=hk, head_dim=d, rope_mode=0, sections=(d // 2, 0, 0), n_sink=6, vision_window=keep - 26, text_window=20)
    s = SideBySide(wl, capacity=max(capacity, keep + 4 + max(sizes)), contiguous=contiguous)
    rng = np.random.default_rng(sum(sizes))
    gid, pos = 0, base
    for rep in range(3):
        for n in sizes:
            s._append(np.arange(gid, gid + n), rng.integers(0, 2, n).astype(np.uint8), (pos + np.arange(n)).astype(np.int32))
            gid, pos = gid + n, pos + n + (gid % 3)
            s.check_metadata()
            s.evict()
            s.check_metadata()
            for layer in range(layers):
                s.check_kv(layer)


# --- one launch each, what the shapes above leave out: more tokens of one ring leaving than the block has threads, three position
# --- axes that differ, positions beyond 2^16, an append that does not fit
@pytest.mark.parametrize("d,hk,vision,leaving", [(64, 1, True, 300), (64, 1, False, 600), (128, 1, True, 257), (64, 2, False, 1000)])
def test_small_caches_evict_more_than_they_keep(d, hk, vision, leaving):
    from harness import SideBySide
    wl = _wl(2, layers=1, q_heads=hk, kv_heads=hk, head_dim=d, rope_mode=0, sections=(d // 2, 0, 0), n_sink=4, vision_window=60, text_window=50)
    s = SideBySide(wl, capacity=leaving + 400)
    rng = np.random.default_rng(leaving)
    gid = 0
    for n, types in ((150, rng.integers(0, 2, 150)), (leaving, np.full(leaving, int(vision))), (40, rng.integers(0, 2, 40)), (leaving, np.full(leaving, int(vision)))):
        s._append(np.arange(gid, gid + n), types.astype(np.uint8), (gid + np.arange(n)).astype(np.int32))
        gid += n
        s.evict()
        s.check_metadata()
        s.check_kv(0)


@pytest.mark.parametrize("d,hk,layers,base", [(64, 1, 1, 0), (64, 2, 2, 0), (128, 1, 1, 70000)])
def test_small_appends_of_three_axes_and_beyond_capacity(d, hk, layers, base):
    from harness import SideBySide
    from paper_2510_09608_b200 import binding
    wl = _wl(2, layers=layers, q_heads=hk, kv_heads=hk, head_dim=d, rope_mode=1, sections=(d // 8, d // 16 * 3, d // 16 * 3), n_sink=6, vision_window=34, text_window=20)
    s = SideBySide(wl, capacity=90)
    rng = np.random.default_rng(d)
    gid, top = 0, base
    for n in (13, 16, 1, 11, 15, 16):
        types = rng.integers(0, 2, n).astype(np.uint8)
        pos = (top + rng.integers(0, 30, (n, 3))).astype(np.int32)          # three axes that differ, not in order
        s._append(np.arange(gid, gid + n), types, pos)
        gid, top = gid + n, top + 30
        s.check_metadata()
        s.evict()
        s.check_metadata()
        for layer in range(layers):
            s.check_kv(layer)
    kept = s.ref.count()
    for n in (16, 16):                                                       # the second one does not fit
        pos = np.repeat((top + np.arange(n, dtype=np.int32))[:, None], 3, axis=1)
        if kept + n <= 90:
            s._append(np.arange(gid, gid + n), np.ones(n, np.uint8), pos)
            gid, top, kept = gid + n, top + n, kept + n
    before = (s.cache.query(), [s.cache.read_kv(l, kept) for l in range(layers)])
    k = torch.ones(layers, 90 - kept + 1, hk, d, dtype=torch.bfloat16, device="cuda")
    n = k.shape[1]
    assert n * layers * hk * d <= 4096                                       # one launch places and writes
    s.cache.append(-1, k, k, torch.ones(n, dtype=torch.uint8, device="cuda"), torch.full((n, 3), top, dtype=torch.int32, device="cuda"))
    after = (s.cache.query(), [s.cache.read_kv(l, kept) for l in range(layers)])
    assert s.cache.status() == binding.ERR_CAPACITY
    assert all(np.array_equal(before[0][key], after[0][key]) for key in ("gids", "pos", "types")) and before[0]["shift_total"] == after[0]["shift_total"]
    assert all(np.array_equal(x, y) for a, b in zip(before[1], after[1]) for x, y in zip(a, b))


def test_small_caches_evict_together():
    """One launch for caches of different windows, one of them with native positions (its keys stay as they are), with more
    leaving one of them than the block has threads."""
    from harness import SideBySide
    from paper_2510_09608_b200 import binding
    windows, natives = [(40, 30), (90, 12), (7, 100)], [False, True, False]
    sides = []
    for i, ((vw, tw), native) in enumerate(zip(windows, natives)):
        wl = _wl(2, layers=1, q_heads=1, kv_heads=1, head_dim=64, rope_mode=0, sections=(32, 0, 0), n_sink=5, vision_window=vw, text_window=tw)
        sides.append(SideBySide(wl, stream=i, capacity=640, contiguous=not native))
    rng = np.random.default_rng(3)
    at = [0] * 3
    for rep, sizes in enumerate([(60, 90, 20), (30, 400, 300), (10, 20, 500), (64, 1, 64)]):
        for i, (s, n) in enumerate(zip(sides, sizes)):
            types = np.ones(n, np.uint8) if n >= 400 else rng.integers(0, 2, n).astype(np.uint8)
            s._append(np.arange(at[i], at[i] + n), types, (at[i] + np.arange(n)).astype(np.int32))
            at[i] += n
        launches = binding.launch_count()
        binding.evict_batched([s.cache for s in sides])
        assert binding.launch_count() == launches + 1
        for s in sides:
            s.rot.evict(s.ref)
            s.check_metadata()
            s.check_kv(0)


def test_a_captured_small_eviction_replayed_with_more_to_evict():
    """The route was chosen when the graph was captured; what leaves when it is replayed is more than fits the lists in shared memory."""
    from harness import SideBySide
    wl = _wl(2, layers=1, q_heads=1, kv_heads=1, head_dim=64, rope_mode=0, sections=(32, 0, 0), n_sink=5, vision_window=90, text_window=60)
    s = SideBySide(wl, capacity=3600)
    rng = np.random.default_rng(9)
    s._append(np.arange(200), rng.integers(0, 2, 200).astype(np.uint8), np.arange(200, dtype=np.int32))
    s.evict()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        s.cache.set_stream(torch.cuda.current_stream())
        s.cache.evict()
    s.cache.set_stream(torch.cuda.current_stream())
    gid = 200
    for n in (30, 3000, 40, 2500):
        s._append(np.arange(gid, gid + n), rng.integers(0, 2, n).astype(np.uint8), (gid + np.arange(n)).astype(np.int32))
        gid += n
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        s.rot.evict(s.ref)
        s.check_metadata()
        s.check_kv(0)


# --- decode: one to three units per warp, a second round, the step to the streaming kernel; one, two and three caches
@pytest.mark.parametrize("d,hq,hk,vw,streams", [
    (128, 28, 4, 100, 1), (64, 5, 1, 40, 1), (128, 8, 8, 4700, 1), (128, 8, 8, 6300, 1), (64, 16, 8, 6300, 1),
    (128, 14, 2, 300, 2), (128, 28, 4, 6200, 2), (64, 4, 1, 700, 3), (128, 28, 4, 3000, 3)])
def test_decode_kernel_choice(d, hq, hk, vw, streams):
    from harness import SideBySide, assert_close, bits_to_dev, dev_to_f64
    from paper_2510_09608_b200 import binding
    wl = _wl(2, layers=1, q_heads=hq, kv_heads=hk, head_dim=d, sections=(d // 8, d // 16 * 3, d // 16 * 3), n_sink=20, vision_window=vw, text_window=30,
             frames=4, grid_h=12, grid_w=13, text_max=9)
    sides = [SideBySide(wl, stream=i) for i in range(streams)]
    for i, s in enumerate(sides):
        for _ in range(1 + vw // 624 + i % 2):
            s.append_chunk()
            s.evict()
    for step in range(2):
        toks = [s.stream.next_decode_token() for s in sides]
        K, V, Q = (np.stack([getattr(s.stream, w)(0, t[0])[0] for s, t in zip(sides, toks)]) for w in "kvq")
        ty = torch.from_numpy(np.concatenate([t[1] for t in toks])).cuda()
        ps = torch.from_numpy(np.ascontiguousarray(np.stack([t[2][0] for t in toks]))).cuda()
        out = dev_to_f64(binding.decode_step_batched([s.cache for s in sides], 0, bits_to_dev(K), bits_to_dev(V), ty, ps, bits_to_dev(Q)))
        for i, (s, t) in enumerate(zip(sides, toks)):
            assert s.cache.status() == binding.OK
            s.ref.append(None, None, t[1], t[2])
            s._give_values_to_ref(0)
            assert_close(s._stats(out[i][None], s.ref.attend(0, Q[i][None], t[2])))
    for s in sides:
        s.check_metadata()
        s.check_kv(0)


# --- projections: a few tokens with weights beyond L2 (512 layers' worth of this size) and within, stages that do not fill,
# --- more rows than one wave of blocks takes; token tiles around multiples of 32, odd numbers of 128-row blocks
@pytest.mark.parametrize("layers,n,in_dim,out_dim", [
    (512, 1, 576, 128), (512, 4, 1088, 384), (512, 2, 3584, 640), (512, 3, 4160, 8448), (512, 1, 128, 1152), (1, 1, 4160, 640),
    (512, 4, 25600, 128),
    (1, 17, 64, 128), (1, 31, 128, 384), (1, 33, 448, 640), (1, 160, 64, 256), (1, 161, 192, 896), (1, 257, 3584, 256), (1, 1400, 128, 1152)])
def test_projection_shapes(layers, n, in_dim, out_dim):
    from harness import bits_to_dev, dev_to_f64
    from oracle import qkv
    from paper_2510_09608_b200 import binding
    rng = np.random.default_rng(n + in_dim)
    A = qkv.to_bf16_bits(rng.standard_normal((n, in_dim)))
    W = qkv.to_bf16_bits(rng.standard_normal((out_dim, in_dim)) / np.sqrt(in_dim))
    c = binding.Cache(layers, 1, 64, 4, 64, 16, 128)
    a, w = bits_to_dev(A), bits_to_dev(W)
    want = qkv.out_project(A, W)
    for _ in range(2):                               # the second call starts while the first one ends
        Y = c.out_proj(a, w)
    assert np.all(np.abs(dev_to_f64(Y) - want) <= 2.0 ** -8 * np.abs(want) + 1e-5 * np.sqrt(in_dim))
    assert c.status() == binding.OK


# --- rows in whole stages, with a shorter last one, all shorter; one to four stages per warp, one to four tokens
@pytest.mark.parametrize("n", [1, 2, 3, 4])
@pytest.mark.parametrize("in_dim,out_dim", [(512, 9088), (2048, 6144), (3584, 2048), (2880, 4096), (4544, 1152), (1344, 4096), (896, 8448), (1280, 640)])
def test_projection_stages(n, in_dim, out_dim):
    test_projection_shapes(512, n, in_dim, out_dim)


# --- one layer's token from host memory, page-locked or not: moved by kernels up to 64 KB, by copies above; the same bits as
# --- from device memory (two layers in turn; all layers of a cache that has one, where the step appends by itself)
@pytest.mark.parametrize("layers", [2, 1])
@pytest.mark.parametrize("d,hq,hk,pinned", [(64, 4, 1, True), (128, 28, 4, True), (128, 28, 4, False), (128, 96, 12, True), (128, 160, 20, False)])
def test_host_decode_steps_of_one_layer(d, hq, hk, pinned, layers):
    from paper_2510_09608_b200 import binding
    rng = np.random.default_rng(hq)
    bits = lambda *shape: torch.from_numpy(rng.standard_normal(shape).astype(np.float32)).to(torch.bfloat16)      # noqa: E731
    keep = (lambda t: t.pin_memory()) if pinned else (lambda t: t)
    dev, host = (binding.Cache(layers, hk, d, 4, 150, 60, 512) for _ in range(2))
    for c in (dev, host):
        c.set_rope(binding.ROPE_1D, 1.0e4)
    k, v = bits(layers, 200, hk, d), bits(layers, 200, hk, d)
    ty, ps = torch.ones(200, dtype=torch.uint8), torch.arange(200, dtype=torch.int32)
    for c in (dev, host):
        c.append(-1, k.cuda(), v.cuda(), ty.cuda(), ps.cuda())
        c.evict()
    for step in range(3):
        for l in (range(2) if layers == 2 else (-1,)):
            k, v, q = bits(1, hk, d), bits(1, hk, d), bits(1, hq, d)
            ty, ps = torch.zeros(1, dtype=torch.uint8), torch.tensor([200 + step], dtype=torch.int32)
            want = dev.decode_step(l, k.cuda(), v.cuda(), ty.cuda(), ps.cuda(), q.cuda())
            out = keep(torch.empty_like(q))
            host.decode_step_host(l, keep(k), keep(v), keep(ty), keep(ps), keep(q), out)
            assert host.status() == binding.OK
            assert torch.equal(out.view(torch.int16), want.cpu().view(torch.int16)), (step, l)


def test_host_prefill_of_large_transfers():
    """All layers of a chunk whose queries are more than the size from which the host waits before it enqueues the copies."""
    from harness import bits_to_dev
    from paper_2510_09608_b200 import binding, streamgen as sg
    wl = _wl(2, layers=4, n_sink=16, vision_window=900, text_window=32, frames=3, grid_h=14, grid_w=14)
    stream = sg.Stream(wl, 0)
    c = binding.Cache(wl.layers, wl.kv_heads, wl.head_dim, wl.n_sink, wl.vision_window, wl.text_window, wl.capacity)
    c.set_rope(wl.rope_mode, wl.rope_base, wl.sections)
    for _ in range(2):
        gids, types, pos = stream.next_chunk()
        K, V, Q = (np.stack([getattr(stream, w)(l, gids) for l in range(wl.layers)]) for w in "kvq")
        ps = torch.from_numpy(np.ascontiguousarray(pos))
        c.append(-1, bits_to_dev(K), bits_to_dev(V), torch.from_numpy(types).cuda(), ps.cuda())
        c.evict()
        assert Q.nbytes >= 16 << 20
        got = torch.empty(Q.shape, dtype=torch.int16).pin_memory()
        c.attend_host(-1, torch.from_numpy(Q.view(np.int16)).pin_memory(), ps.pin_memory(), got)
        want = torch.stack([c.attend(l, bits_to_dev(Q[l]), ps.cuda()) for l in range(wl.layers)])
        assert torch.equal(got, want.view(torch.int16).cpu())
        assert c.status() == binding.OK


def test_few_token_projection_gives_up_and_recovers():
    """Every wait of the projection for a few tokens made to run out: the status appears, the kernel returns, and with the
    limit restored it computes."""
    from harness import bits_to_dev, dev_to_f64
    from oracle import qkv
    from paper_2510_09608_b200 import binding
    rng = np.random.default_rng(5)
    A, W = qkv.to_bf16_bits(rng.standard_normal((2, 1088))), qkv.to_bf16_bits(rng.standard_normal((384, 1088)) / 33)
    c = binding.Cache(512, 1, 64, 4, 64, 16, 128)
    a, w = bits_to_dev(A), bits_to_dev(W)
    c.debug_set_wait_limit(0)
    c.out_proj(a, w)
    assert c.status() == binding.ERR_TIMEOUT
    c.debug_set_wait_limit(1 << 20)
    want = qkv.out_project(A, W)
    assert np.all(np.abs(dev_to_f64(c.out_proj(a, w)) - want) <= 2.0 ** -8 * np.abs(want) + 1e-3)


# --- one token's rows at any element of an array and its output at any word: per-layer kernel (one cache, two), streaming
# --- kernel (three rounds of keys, many caches); the same bits as from aligned buffers
@pytest.mark.parametrize("d,hq,hk,kept,streams", [(128, 28, 4, 300, 1), (64, 5, 1, 90, 1), (128, 8, 8, 11000, 1), (128, 14, 2, 300, 2), (64, 16, 8, 200, 4)])
def test_decode_inputs_at_any_element(d, hq, hk, kept, streams):
    from paper_2510_09608_b200 import binding

    def shifted(t, by):
        flat = torch.zeros(t.numel() + 8, dtype=t.dtype, device="cuda")
        flat[by:by + t.numel()] = t.flatten()
        return flat[by:by + t.numel()].view(t.shape)

    def run(by):
        gen = torch.Generator(device="cuda").manual_seed(kept)
        normal = lambda *shape: torch.randn(*shape, generator=gen, device="cuda", dtype=torch.bfloat16)      # noqa: E731
        caches = [binding.Cache(1, hk, d, 4, kept, 60, kept + 200) for _ in range(streams)]
        for c in caches:
            c.append(-1, normal(1, kept, hk, d), normal(1, kept, hk, d), torch.ones(kept, dtype=torch.uint8, device="cuda"),
                     torch.arange(kept, dtype=torch.int32, device="cuda"))
        outs = []
        for t in range(3):
            k, v, q = (shifted(normal(streams, h, d), b) for h, b in ((hk, by), (hk, 3 * by), (hq, by)))
            ty = torch.zeros(streams, dtype=torch.uint8, device="cuda")
            ps = torch.full((streams,), kept + t, dtype=torch.int32, device="cuda")
            out = shifted(torch.zeros_like(q), 2 * by)
            if streams == 1:
                caches[0].decode_step(0, k, v, ty, ps, q, out)
            else:
                binding.decode_step_batched(caches, 0, k, v, ty, ps, q, out)
            outs.append(out.clone())
        assert all(c.status() == binding.OK for c in caches)
        return torch.stack(outs).view(torch.int16)

    want = run(0)
    assert torch.equal(run(1), want) and want.any()


# --- decode steps whose launch appends the token itself (one cache or several of one layer; beside them all layers at once): tokens that
# --- open pages of either ring and of the sinks, vision among text, evictions in between, both kernels, and a cache that is full
@pytest.mark.parametrize("d,hq,hk,layers,streams,rope_1d,sink_any,fill", [
    (64, 4, 1, 1, 1, True, False, 60), (128, 28, 4, 1, 1, False, False, 500), (128, 8, 4, 3, 1, False, True, 100), (64, 16, 8, 1, 4, True, True, 250),
    (128, 14, 2, 1, 2, False, False, 130), (128, 28, 4, 1, 5, False, False, 300)])
def test_decode_steps_that_append_by_themselves(d, hq, hk, layers, streams, rope_1d, sink_any, fill):
    from harness import SideBySide, assert_close, bits_to_dev, dev_to_f64
    from paper_2510_09608_b200 import binding
    half = d // 2
    wl = _wl(2, layers=layers, q_heads=hq, kv_heads=hk, head_dim=d, rope_mode=0 if rope_1d else 1,
             sections=(half, 0, 0) if rope_1d else (half // 4, 3 * half // 8, 3 * half // 8), n_sink=130, vision_window=fill, text_window=140)
    rng = np.random.default_rng(fill)
    sides = [SideBySide(wl, stream=i, capacity=130 + fill + 140 + 160, sink_any=sink_any) for i in range(streams)]
    at = [0] * streams                                           # next ordinal, and its native position
    shaped = lambda p: np.asarray(p, np.int32) if rope_1d else np.repeat(np.asarray(p, np.int32)[:, None], 3, axis=1)     # noqa: E731
    for i, s in enumerate(sides):
        n = fill + 17 * i
        s._append(np.arange(n), rng.integers(0, 2, n).astype(np.uint8), shaped(np.arange(n)))
        at[i] = n
    before = binding.launch_count()
    steps = 290
    for step in range(steps):
        types = rng.integers(0, 2, streams).astype(np.uint8)
        pos = np.stack([shaped([at[i]]) for i in range(streams)])          # [streams, 1(, 3)]
        ty, ps = torch.from_numpy(types).cuda(), torch.from_numpy(pos).cuda()
        gids = [np.arange(at[i], at[i] + 1) for i in range(streams)]
        rows = lambda what: np.stack([np.stack([getattr(s.stream, what)(l, g) for s, g in zip(sides, gids)]) for l in range(layers)])  # noqa: E731  [layers, streams, 1, heads, d]
        K, V, Q = (bits_to_dev(rows(w)) for w in "kvq")
        if streams > 1:
            out = binding.decode_step_batched([s.cache for s in sides], 0, K[0, :, 0].contiguous(), V[0, :, 0].contiguous(), ty, ps[:, 0].contiguous(), Q[0, :, 0].contiguous())[None, :, None]
        elif layers > 1:
            out = sides[0].cache.decode_step(-1, K[:, 0].contiguous(), V[:, 0].contiguous(), ty, ps[0], Q[:, 0].contiguous())[:, None]
        else:
            out = sides[0].cache.decode_step(0, K[0, 0], V[0, 0], ty, ps[0], Q[0, 0])[None, None]
        for i, s in enumerate(sides):
            s.ref.append(None, None, types[i:i + 1], pos[i])
            at[i] += 1
        if step % 41 == 0 or step == steps - 1:
            for i, s in enumerate(sides):
                s.check_metadata()
                for l in {0, layers - 1}:
                    s._give_values_to_ref(l)
                    assert_close(s._stats(dev_to_f64(out)[l, i], s.ref.attend(l, s.stream.q(l, gids[i]), pos[i])))
        if step % 97 == 96:
            for s in sides:
                s.evict()
                s.check_metadata()
    if streams == 1 and layers == 1:
        assert binding.launch_count() - before <= steps + 2 * (steps // 97)     # one launch a step
    for s in sides:
        for l in {0, layers - 1}:
            s.check_kv(l)
    s = sides[0]                                                 # until it is full: the token is dropped, the status says so, nothing else moves
    kept = len(s.cache.query()["gids"])
    K, V, Q = (bits_to_dev(np.stack([getattr(s.stream, w)(l, np.arange(1)) for l in range(layers)])) for w in "kvq")
    ty = torch.zeros(1, dtype=torch.uint8, device="cuda")
    for _ in range(130 + fill + 140 + 160 - kept + 3):
        s.cache.decode_step(-1, K, V, ty, torch.from_numpy(shaped([at[0]])).cuda(), Q)
        at[0] += 1
    assert s.cache.status() == binding.ERR_CAPACITY
    assert len(s.cache.query()["gids"]) == 130 + fill + 140 + 160


def test_decode_alternating_single_and_batched():
    """The same caches decode by themselves, in pairs and all together in turn: the per-layer kernel writes its tagged records
    with 37 splits, then 18, the streaming kernel its own scratch with 9, and none may take another's leftovers for its own."""
    from harness import SideBySide, assert_close, bits_to_dev, dev_to_f64
    from paper_2510_09608_b200 import binding
    wl = _wl(2, layers=1, n_sink=20, vision_window=1500, text_window=30, frames=4, grid_h=8, grid_w=8, text_max=9)
    sides = [SideBySide(wl, stream=i) for i in range(4)]
    for s in sides:
        for _ in range(7):
            s.append_chunk()
            s.evict()
    for group in (1, 2, 4, 2, 1, 1, 4, 1, 2):
        for at in range(0, 4, group):
            part = sides[at:at + group]
            toks = [s.stream.next_decode_token() for s in part]
            K, V, Q = (np.stack([getattr(s.stream, w)(0, t[0])[0] for s, t in zip(part, toks)]) for w in "kvq")
            ty = torch.from_numpy(np.concatenate([t[1] for t in toks])).cuda()
            ps = torch.from_numpy(np.ascontiguousarray(np.stack([t[2][0] for t in toks]))).cuda()
            if group == 1:
                out = part[0].cache.decode_step(0, bits_to_dev(K), bits_to_dev(V), ty, ps, bits_to_dev(Q))
            else:
                out = binding.decode_step_batched([s.cache for s in part], 0, bits_to_dev(K), bits_to_dev(V), ty, ps, bits_to_dev(Q))
            out = dev_to_f64(out)
            for i, (s, t) in enumerate(zip(part, toks)):
                assert s.cache.status() == binding.OK
                s.ref.append(None, None, t[1], t[2])
                s._give_values_to_ref(0)
                assert_close(s._stats(out[i][None], s.ref.attend(0, Q[i][None], t[2])))
