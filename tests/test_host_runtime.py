"""The library's host side (argument checks, routes, failing calls) on a stand-in for the CUDA runtime: no GPU, nothing runs."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# What every test program starts with: the library over the stand-in, a one-stream cache, and short calls.  Pointers are
# made-up numbers: the host side never follows them.
PRELUDE = """
import ctypes as C, sys
fake = C.CDLL(sys.argv[1], mode=C.RTLD_GLOBAL)
lib = C.CDLL(sys.argv[2])
fake.fake_log.restype = C.c_char_p
fake.fake_alloc_limit.argtypes = [C.c_size_t]
OK, ARG, CAPACITY, ORDER, CUDA = 0, -1, -2, -3, -4
P = 1 << 20
vp = C.c_void_p

def new(layers=1, hk=4, d=128, sink=4, vw=1000, tw=100, capacity=1500):
    h = vp()
    assert lib.svlm_cache_create(C.byref(h), layers, hk, d, sink, vw, tw, capacity) == OK
    return h

def append(c, n, layer=0, K=P, V=P):
    return lib.svlm_cache_append(c, layer, vp(K), vp(V), vp(P), vp(P), n)

def attend(c, n, hq=28, layer=0, Q=P, out=P, pos=P):
    return lib.svlm_attend(c, layer, vp(Q), vp(pos), n, hq, vp(out))

def step(c, hq=28, layer=0, K=P, V=P, Q=P, out=P):
    return lib.svlm_decode_step(c, layer, vp(K), vp(V), vp(P), vp(P), vp(Q), hq, vp(out))

def arr(caches):
    return (vp * len(caches))(*caches)

def ran():
    return fake.fake_log().decode().splitlines()
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    from paper_2510_09608_b200 import build
    fake = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.check_call(["g++", "-shared", "-fPIC", "-O1", "-I/usr/local/cuda/include", "-o", fake, os.path.join(ROOT, "tests", "fake_cudart.cpp")])
    lib = build.build()

    def run(body):
        res = subprocess.run([sys.executable, "-c", PRELUDE + body, fake, lib], capture_output=True, text=True, timeout=120)
        assert res.returncode == 0, res.stdout + res.stderr
        return res.stdout
    return run


def test_alignment_of_device_pointers(host):
    """One token's rows may begin at any element and its output at any word; chunks want 16 bytes; what is refused launches nothing."""
    host("""
c = new()
assert append(c, 40) == OK
ran()
for kw in (dict(K=P + 8), dict(V=P + 2)):
    assert append(c, 40, **kw) == ARG
for kw in (dict(Q=P + 2), dict(out=P + 8), dict(pos=P + 2)):
    assert attend(c, 40, **kw) == ARG
for kw in (dict(Q=P + 1), dict(out=P + 2), dict(K=P + 3), dict(V=P + 1)):
    assert step(c, **kw) == ARG
assert attend(c, 1, out=P + 2) == ARG and attend(c, 1, Q=P + 1) == ARG
two = arr([c, new()])
assert append(two[1], 40) == OK
ran()
call = lambda Q, out: lib.svlm_decode_step_batched(two, 2, 0, vp(P), vp(P), vp(P), vp(P), vp(Q), 28, vp(out))
assert call(P + 1, P) == ARG and call(P, P + 2) == ARG
n = (C.c_int32 * 2)(3, 4)
assert lib.svlm_attend_batched_varlen(two, 2, 0, vp(P + 2), vp(P), n, 28, vp(P)) == ARG
assert lib.svlm_attend_decode_noalloc(c, 0, vp(P), vp(P), 28, vp(P + 2)) == ARG
assert ran() == []
assert step(c, K=P + 2, V=P + 6, Q=P + 2, out=P + 4) == OK and attend(c, 1, Q=P + 2, out=P + 4) == OK
assert call(P + 2, P + 4) == OK
assert lib.svlm_attend_decode_noalloc(c, 0, vp(P + 2), vp(P), 28, vp(P + 4)) == OK
wide = new(hk=1, capacity=70000)                    # more pages than the fast kernels' lists: the general kernel, element by element
assert append(wide, 40) == OK and attend(wide, 40, hq=4, Q=P + 2, out=P + 2) == OK and attend(wide, 1, hq=9, Q=P + 2, out=P + 2) == OK
""")


def test_a_failed_metadata_launch_ends_the_call(host):
    """Nothing that relies on the metadata is launched behind it, the host's counts stay, and the error is the call's alone."""
    host("""
c, d = new(layers=2), new(layers=2)
both = arr([c, d])
qkv = lambda: lib.svlm_qkv_append(c, 0, vp(P), vp(P), 128, 28, vp(P), vp(P), 40, vp(P))
steps = lambda: lib.svlm_decode_step_batched(both, 2, 0, vp(P), vp(P), vp(P), vp(P), vp(P), 28, vp(P))
for x in (c, d):
    assert append(x, 40) == OK
ran()
fake.fake_fail(b"append_meta")
for call in (lambda: append(c, 40), lambda: append(c, 40, layer=-1), qkv, lambda: step(c), steps):
    assert call() == CUDA and ran() == [] and fake.cudaGetLastError() == 0
    assert attend(c, 41) == ORDER and append(c, 40, layer=1) == OK       # the host still reckons with the first 40 tokens
    ran()
fake.fake_fail(b"evict_meta")
assert lib.svlm_cache_evict(c) == CUDA and lib.svlm_cache_evict_batched(both, 2) == CUDA and ran() == [] and fake.cudaGetLastError() == 0
fake.fake_fail(b"")
assert append(c, 40) == OK and steps() == OK and lib.svlm_cache_evict(c) == OK
""")


def test_a_failed_launch_of_a_call_that_is_one_launch_ends_it(host):
    """Steps that append by themselves (one cache by either decode kernel, a batch), appends and evictions of small caches: the host's
    counts are what they were, nothing else is launched, and the next call does what it would have done."""
    host("""
def fails(kernel, calls, caches, n):
    fake.fake_fail(kernel)
    for call in calls:
        ran()
        assert call() == CUDA and ran() == [] and fake.cudaGetLastError() == 0, kernel
        fake.fake_fail(b"")
        for c in caches:
            assert attend(c, n + 1, hq=8) == ORDER and attend(c, n, hq=8) == OK      # n tokens so far
        fake.fake_fail(kernel)
    fake.fake_fail(b"")
near = new(hk=8)                                          # one layer: the per-layer kernel, over more keys the streaming one
far = new(hk=8, vw=26000, tw=100, capacity=26300)
four = [new(hk=8) for _ in range(4)]
for c in [near, far] + four:
    assert append(c, 40) == OK
for _ in range(20):
    assert append(far, 1300) == OK
batched = lambda cs: lib.svlm_decode_step_batched(arr(cs), len(cs), 0, vp(P), vp(P), vp(P), vp(P), vp(P), 8, vp(P))
fails(b"decode_layer", [lambda: step(near, hq=8), lambda: step(near, hq=8, layer=-1), lambda: batched([near])], [near], 40)
fails(b"decode_stream", [lambda: step(far, hq=8)], [far], 26040)
fails(b"decode_stream", [lambda: batched(four)], four, 40)
for call, name in ((lambda: step(near, hq=8), "decode_layer"), (lambda: step(far, hq=8), "decode_stream"), (lambda: batched(four), "decode_stream")):
    ran()
    assert call() == OK
    got = ran()
    assert len(got) == 1 and name in got[0], got
assert attend(near, 42, hq=8) == ORDER and attend(near, 41, hq=8) == OK
small = [new(hk=1, d=64, vw=120, tw=70, capacity=400) for _ in range(2)]
for c in small:
    ran()
    assert append(c, 40) == OK
    got = ran()
    assert len(got) == 1 and "append_meta_write" in got[0], got
fails(b"append_meta_write", [lambda: append(small[0], 40), lambda: append(small[0], 40, layer=-1)], small, 40)
fails(b"evict_meta", [lambda: lib.svlm_cache_evict(small[0]), lambda: lib.svlm_cache_evict_batched(arr(small), 2)], small, 40)
""")


def test_a_captured_call_is_reckoned_with_full_windows(host):
    """A graph captured while the windows fill is replayed when they are full: the kernels are chosen for that, and so they are
    for plain calls of the same cache afterwards, whose appends the host may not have seen."""
    host("""
def kernels(call):
    ran()
    assert call() == OK
    return [l.split()[0] for l in ran()]
small = lambda names: any("prefill_small" in n for n in names)
layer = lambda names: any("decode_layer" in n for n in names)
big = dict(layers=6, hk=8, vw=12000, tw=500, capacity=13000)
for calls in (lambda c: attend(c, 133, hq=32), lambda c: lib.svlm_attend_batched_varlen(arr([c]), 1, 0, vp(P), vp(P), (C.c_int32 * 1)(133), 32, vp(P))):
    c = new(**big)
    assert append(c, 133) == OK and small(kernels(lambda: calls(c)))
    fake.fake_capturing(1)
    assert not small(kernels(lambda: calls(c)))
    fake.fake_capturing(0)
    assert not small(kernels(lambda: calls(c)))
    full = new(**big)                                    # what an ordinary stream takes when its windows are full
    for _ in range(120):
        assert append(full, 133) == OK and lib.svlm_cache_evict(full) == OK
    assert not small(kernels(lambda: calls(full)))
c = new(**big)
assert append(c, 133) == OK and layer(kernels(lambda: step(c, hq=32)))
fake.fake_capturing(1)
assert append(c, 133) == OK                              # captured: the host does not see when it runs
fake.fake_capturing(0)
assert not layer(kernels(lambda: step(c, hq=32))) and not layer(kernels(lambda: step(full, hq=32)))
""")


@pytest.mark.parametrize("layers,kv_heads,d,keys,kernel", [
    (1, 8, 128, 10000, "layer"), (1, 8, 128, 23000, "layer"), (1, 8, 128, 26000, "stream"), (2, 8, 128, 10500, "layer"), (2, 8, 128, 13000, "stream"),
    (6, 8, 128, 5000, "layer"), (6, 8, 128, 10500, "stream"), (28, 4, 128, 20000, "layer"), (28, 8, 64, 20000, "layer")])
def test_decode_kernel_of_one_stream(host, layers, kv_heads, d, keys, kernel):
    """Few thread blocks per KV head and more than two rounds of keys: the streaming kernel, unless the keys stay in L2."""
    host(f"""
c = new(layers={layers}, hk={kv_heads}, d={d}, vw={keys}, tw=100, capacity={keys} + 300)
assert append(c, {keys}) == OK
ran()
assert step(c, hq={kv_heads}) == OK and "decode_{kernel}" in "".join(ran())
""")


@pytest.mark.parametrize("layers,in_dim,out_dim,n,kernel", [
    (1, 64, 128, 1, "mma"), (1, 1792, 512, 4, "mma"), (1, 1856, 512, 1, "few"), (1, 3584, 2304, 4, "few"), (1, 3584, 2432, 4, "mma"), (1, 2048, 6144, 1, "few"),
    (1, 3648, 4608, 1, "few"), (1, 3584, 4608, 5, "mma"), (28, 3584, 4608, 1, "few"), (1, 25600, 128, 4, "mma")])
def test_projection_kernel_of_a_few_tokens(host, layers, in_dim, out_dim, n, kernel):
    host(f"""
c = new(layers={layers}, capacity=1500 if {layers} == 1 else 200)
assert lib.svlm_out_proj(c, vp(P), vp(P), {in_dim}, {out_dim}, {n}, vp(P)) == OK
assert "gemv_{kernel}" in "".join(ran())
""")


@pytest.mark.parametrize("in_dim,form", [(512, 0), (3584, 0), (8192, 0), (2304, 1), (4160, 1), (5440, 1), (64, 2), (576, 2), (1280, 2), (1344, 2), (2688, 2)])
def test_projection_form_of_a_few_tokens(host, in_dim, form):
    """Rows in stages that are all of one length, all but the last, or all shorter: a kernel each."""
    host(f"""
c = new(layers=800, hk=1, d=64, vw=64, tw=16, capacity=128)
assert lib.svlm_out_proj(c, vp(P), vp(P), {in_dim}, 4096, 1, vp(P)) == OK
assert "gemv_few_kernelILi{form}E" in "".join(ran())
""")


PLAN_PROGRAM = r"""
#include <cassert>
#include <cstdio>
#include "svlm_prefill_plan.h"

static SvlmAttendBatch batch(int kv_heads) { SvlmAttendBatch b{}; b.n_caches = 1; b.kv_heads = kv_heads; return b; }

// A cut unit's pieces are counted alike by all that hold one, and its columns are shared out once among those that end in it.
static void check_cut_units(const PfPlan& plan, int grid, int nt, int blocks) {
    for (int t = 0; t < nt; ++t) {
        const int u0 = t * PF_FRAC, u1 = u0 + PF_FRAC;
        int pieces = 0, ends = 0;
        unsigned shared = 0;
        for (int k = 0; k < grid; ++k) {
            const bool here = plan.x[k] < plan.x[k + 1] && plan.x[k] < u1 && plan.x[k + 1] > u0;
            pieces += here;
            ends += here && plan.x[k + 1] <= u1;
        }
        if (pieces < 2) continue;
        for (int k = 0; k < grid; ++k) {
            if (!(plan.x[k] < plan.x[k + 1] && plan.x[k] < u1 && plan.x[k + 1] > u0)) continue;
            const PfCut c = pf_cut(plan, t, k, blocks);
            assert(c.pieces == pieces && (c.sharers > 0) == (blocks == 8 && ends > 1) && plan.x[c.first] <= u0 && plan.x[c.first] < plan.x[c.first + 1] && plan.x[c.last + 1] >= u1);
            assert(!(c.mine & shared) && (!c.mine || plan.x[k + 1] <= u1));
            shared |= c.mine;
        }
        assert(shared == (blocks == 8 && ends > 1 ? 255u : 0u));      // heads of 64, or one that ends in it: the last one merges all
    }
}

int main() {
    PfPlanMemo& memo = pf_plan_memo();
    SvlmAttendBatch b = batch(4);
    SvlmPrefillLoad held[SVLM_MAX_BATCH] = {{76, 8704}};
    // streams served in turn, layer after layer: a split per size, not per call
    for (int layer = 0; layer < 28; ++layer)
        for (int stream = 0; stream < 8; ++stream) pf_plan(b, 1, 512 + stream, 7, held, 148, true);
    assert(memo.made == 8);
    for (int layer = 0; layer < 28; ++layer) pf_plan(b, 1, 524, 7, held, 148, true);      // more streams than entries: still right
    for (int n = 2; n < 400; n += 13) pf_plan(b, 1, n, 7, held, 148, true);
    // every page fraction of every unit is dealt out once, in order
    long long checked = 0;
    unsigned cuts = 2166136261u;
    for (int kv_heads : {1, 4, 8})
        for (int G : {1, 4, 7})
            for (int n : {2, 37, 256, 531, 4133})
                for (int pages : {1, 12, 76, 512})
                    for (int layers : {1, 28})
                        for (int cut : {0, 1}) {
                            b = batch(kv_heads);
                            held[0] = {pages, pages * 128};
                            const PfPlanned& p = pf_plan(b, layers, n, G, held, 148, cut != 0);
                            const int nt = p.plan.units - p.plan.tail;
                            assert(p.grid >= 1 && p.grid <= 148 && p.plan.rounds * p.grid == p.plan.tail && nt >= 0 && nt < 2 * PF_MAX_CTAS);
                            assert(p.plan.units == layers * kv_heads * ((n * G + PF_ROWS - 1) / PF_ROWS));
                            assert(p.plan.x[0] == 0 && p.plan.x[p.grid] == nt * PF_FRAC);
                            for (int i = 0; i < p.grid; ++i) {
                                assert(p.plan.x[i] <= p.plan.x[i + 1]);
                                if (!cut) assert(p.plan.x[i] % PF_FRAC == 0);
                            }
                            for (int i = 0; i <= p.grid; ++i) cuts = (cuts ^ p.plan.x[i]) * 16777619u;
                            for (int blocks : {4, 8}) check_cut_units(p.plan, p.grid, nt, blocks);
                            ++checked;
                        }
    std::printf("%lld %u\n", checked, cuts);
}
"""


def test_chunk_prefill_work_split(tmp_path):
    """The host's work split: remembered by sizes alone, complete, and with the cuts where they have been: a row's weights are rounded
    against the reference maximum of its piece, so outputs change in their last places with the cuts."""
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(PLAN_PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I/usr/local/cuda/include", "-I" + os.path.join(ROOT, "paper_2510_09608_b200", "csrc"),
                           "-o", str(exe), str(src)])
    assert subprocess.check_output([str(exe)], text=True).strip() == f"{3 * 3 * 5 * 4 * 2 * 2} 3026906603"


def test_a_cache_that_fits_without_the_scratch_for_cut_units(host):
    """Memory for the cache but not for the slots of cut units: it is created, and its chunks take whole units."""
    host("""
def blocks(c):
    assert append(c, 300) == OK
    for _ in range(4):
        assert append(c, 250) == OK
    ran()
    assert attend(c, 250) == OK
    name, grid, _ = ran()[-1].split()
    assert "prefill_kernel" in name
    return int(grid.split(",")[0])
size = dict(hk=4, vw=2000, tw=100, capacity=2400)
assert blocks(new(**size)) > 60                     # 28 units of 256 rows, cut in pieces
fake.fake_alloc_limit(20 << 20)
assert blocks(new(**size)) == 28
fake.fake_alloc_limit(1 << 20)
assert lib.svlm_cache_create(C.byref(vp()), 1, 4, 128, 4, 2000, 100, 2400) == -6 and fake.cudaGetLastError() == 0
""")


def test_shapes_of_other_tests_take_the_kernels_they_name(host):
    """The give-up tests (8 pages, 28/4 heads of 128; four caches) and the smoke test's two chunk shapes."""
    host("""
mk = lambda: new(sink=16, vw=192, tw=40, capacity=400)
caches = [mk() for _ in range(4)]
for c in caches:
    assert append(c, 248) == OK
ran()
assert attend(caches[0], 70) == OK and "prefill_small" in ran()[-1]
assert attend(caches[0], 1) == OK and "decode_layer" in ran()[-1]
both = lambda n: lib.svlm_attend_batched(arr(caches[:n]), n, 0, vp(P), vp(P), 1, 28, vp(P))
assert both(2) == OK and "decode_layer" in ran()[-1]
assert both(4) == OK and "decode_stream" in ran()[-1]
for vw, tw, n, kernel in ((512, 64, 130, "prefill_small"), (1536, 128, 520, "14prefill_kernel")):
    c = new(layers=2, sink=32, vw=vw, tw=tw, capacity=vw + tw + n + 40)
    assert append(c, n) == OK and append(c, vw + tw + 32 - n) == OK and append(c, n) == OK and lib.svlm_cache_evict(c) == OK
    ran()
    assert attend(c, n) == OK and kernel in ran()[-1], kernel
""")


def test_evictions_of_many_tokens_take_two_launches(host):
    """One launch serves a small cache's eviction with few threads, which also walk over all tokens that leave: few of them only."""
    host("""
small = dict(layers=1, hk=1, d=64, sink=4, vw=120, tw=70, capacity=5000)
def evicts(c, batch=None):
    ran()
    assert (lib.svlm_cache_evict_batched(arr(batch), len(batch)) if batch else lib.svlm_cache_evict(c)) == OK
    return [l.split()[0] for l in ran()]
one = lambda names: len(names) == 1 and "evict_meta" in names[0]
two = lambda names: len(names) == 2 and "evict_meta" in names[0] and "evict_rotate" in names[1]
c, d = new(**small), new(**small)
for n, kernels in ((194, one), (1024, one), (30, one), (1025, two), (4608, two), (1024, one)):
    assert append(c, n, layer=-1) == OK
    assert kernels(evicts(c)), n
for n, kernels in ((1024, one), (1025, two)):                # of a batch: by the cache that has most to lose
    assert append(c, 40, layer=-1) == OK and append(d, n, layer=-1) == OK
    if n == 1024:
        assert append(d, 194, layer=-1) == OK                # (the windows were empty)
    assert kernels(evicts(None, [c, d])), n
""")


def test_which_host_buffers_the_kernels_read_in_place(host):
    """All layers of a token from mapped host memory: the decode launch reads them where they are, one of each for all the thread
    blocks that want them.  One layer goes through device memory, also when it is all that the cache has."""
    host("""
fake.fake_mapped(1)
buf = (C.c_char * (1 << 16))()
at = vp(C.addressof(buf) + 63 & ~63)
def kernels(layers, layer):
    c = new(layers=layers)
    assert append(c, 40, layer=-1) == OK
    ran()
    assert lib.svlm_decode_step_host(c, layer, at, at, at, at, at, 28, at) == OK
    return " ".join(l.split()[0] for l in ran())
deep = kernels(3, -1)
assert "host_in" not in deep and "append_meta" in deep and "decode" in deep
for layers, layer in ((3, 0), (1, 0), (1, -1)):
    assert "host_in" in kernels(layers, layer), (layers, layer)
""")


def test_when_an_output_from_host_memory_waits_for_the_next_queries(host):
    """All layers of a chunk in one call: an output waits for the next layer's queries where that saves more, over the layers, than the one
    copy that it makes the last output later."""
    host("""
buf = vp(C.addressof((C.c_char * (120 << 20)).from_buffer(mem := bytearray(120 << 20))))
def waits(layers, n, kept, hq, hk, d):
    c = new(layers=layers, hk=hk, d=d, vw=kept, tw=100, capacity=kept + 100)
    assert append(c, kept, layer=-1) == OK
    fake.fake_waits()
    assert lib.svlm_attend_host(c, -1, buf, buf, n, hq, buf) == OK
    early = layers * n * hq * d * 2 < 16 << 20               # (the copies wait for earlier work by an event)
    extra = fake.fake_waits() - 2 * layers - early
    assert extra in (0, layers - 1)
    lib.svlm_cache_destroy(c)
    return extra > 0
big, small = (28, 4, 128), (4, 1, 64)
for n, kept, shape, first in ((2000, 2000, big, 7), (2000, 8192, big, 4), (1000, 1024, big, 5), (524, 1024, big, 3), (266, 1024, big, None), (524, 8192, big, 2),
                              (150, 1024, big, None), (16, 1024, big, None), (524, 1024, (16, 8, 64), None), (2000, 2000, small, None)):
    for layers in range(2, 9):
        if layers * n * shape[0] * shape[2] * 2 < 110 << 20:
            assert waits(layers, n, kept, *shape) == (first is not None and layers >= first), (n, kept, shape, layers)
""")


def test_which_weights_of_a_chunk_are_read_once(host):
    """Weights that stay in L2 from pass to pass keep their place there, unless the chunk is long; where tiles read them again, always."""
    host("""
def once(layers, hidden, out, n):
    c = new(layers=layers, capacity=1500)
    assert lib.svlm_out_proj(c, vp(P), vp(P), hidden, out, n, vp(P)) == OK
    launched = "".join(ran())
    lib.svlm_cache_destroy(c)
    forms = [form for form in (0, 1) if f"qkv_append_kernelILb{form}E" in launched]
    assert len(forms) == 1
    return forms[0]
for layers, hidden, out, n, want in ((4, 1024, 3072, 20, 0), (4, 1024, 3072, 159, 0), (4, 1024, 3072, 160, 1), (3, 2048, 2560, 133, 0), (4, 2048, 2560, 20, 1),
                                     (1, 3584, 4608, 133, 0), (1, 3584, 4608, 524, 1), (2, 3584, 3584, 20, 1), (28, 3584, 3584, 531, 1), (28, 3584, 4608, 4133, 0)):
    assert once(layers, hidden, out, n) == want, (layers, hidden, out, n)
""")
