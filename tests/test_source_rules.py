"""Rules that the compiler does not enforce, checked on the kernels' source."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_09608_b200", "csrc")


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def test_only_constants_take_the_read_only_path():
    """Kernels start while the one before them still runs (programmatic dependent launch), so what an earlier kernel of the
    stream may write (inputs, positions, metadata) is loaded by svlm_ptx::ld_in and ld_l2, which stay behind the wait and are
    coherent.  The read-only path (__ldg, const __restrict__) is for the rotation table and the projections' weights."""
    constants = {"tab", "p", "wp"}      # p, wp: rows of W (svlm_gemv.cu)
    for name in sorted(os.listdir(CSRC)):
        src = _source(name)
        if "pdl_wait" not in src and name != "svlm_rope.cuh":
            continue
        used = set(re.findall(r"__ld(?:g|cg|ca|cs)\(\s*&?\s*(\w+)", src))
        assert used <= constants, (name, used - constants)
        restricted = set(re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", src))
        assert restricted <= {"tab", "W"}, (name, restricted)


def test_only_weights_take_the_inline_read_only_load():
    """The same for ld.global.nc in inline assembly: one function has it, and what it is given are rows of W."""
    inline = [(name, src) for name in sorted(os.listdir(CSRC)) for src in [_source(name)] if re.search(r"ld\.global(\.\w+)*\.nc", src)]
    assert [name for name, _ in inline] == ["svlm_gemv.cu"]
    src = inline[0][1]
    body = re.search(r"uint4 ld_weights\(const uint4\* p, .*?\n\}", src, flags=re.S).group(0)
    assert len(re.findall(r"ld\.global(?:\.\w+)*\.nc", src)) == len(re.findall(r"ld\.global(?:\.\w+)*\.nc", body)) == 1
    calls = re.findall(r"ld_weights\((?!const uint4\*)\s*(\w+)", src)
    assert calls and set(calls) == {"p"} and len(re.findall(r"const uint4\* p = reinterpret_cast<const uint4\*>\(W \+", src)) == 1


def test_waits_for_tensor_memory_name_what_was_loaded():
    """tcgen05.ld fills its registers when the wait behind it is over.  Two volatile statements stay in order, but arithmetic on the
    registers is no such statement: only the wait's naming them keeps it behind."""
    loads = waits = 0
    for name in sorted(os.listdir(CSRC)):
        src = _source(name)
        if name == "svlm_tc.cuh":
            body = re.search(r"void tmem_wait_ld\(float\* v\) \{(.*?)\n\}", src, flags=re.S).group(1)
            assert body.index("tcgen05.wait::ld") < body.index('"+f"(v[i])') and src.count("tcgen05.wait::ld") == 1
            continue
        assert "tcgen05.ld" not in src and "tcgen05.wait::ld" not in src, name
        # between a wait and the one before it: the loads it waits for, and it names as many registers as they fill
        for part in re.split(r"(?<=;)", src):
            if m := re.search(r"\btmem_ld(\d+)\(", part):
                loads += int(m.group(1))
            if re.search(r"\btmem_wait_ld\b", part):
                waits += int(re.search(r"tmem_wait_ld<(\d+)>\(\w", part).group(1))
        assert loads == waits, (name, loads, waits)
    assert loads > 0


def test_what_a_chunk_prefill_block_keeps_of_a_cache_is_written_behind_the_barrier():
    """Between units all threads read what is known of the cache while thread 0 replaces the segment's own fields: the two sets are
    disjoint, and the first one is written behind the barrier that follows the reads."""
    src = _source("svlm_prefill_sm100.cu")
    at = src.index("rows.ci != gr.known")
    known = src[src.index("} else {", at):src.index("rot.load_pos", at)]
    read = set(re.findall(r"= gr\.([\w.]+)", known))
    barrier = src.index("bar_sync(BAR_WG + g, 128);", at)
    assert len(read) == 5
    written_before = set(re.findall(r"gr\.(\w+)(?:\[[^]]*\])? = ", src[at:barrier]))
    written_behind = set(re.findall(r"gr\.(\w+)(?:\[[^]]*\])? = ", src[barrier:src.index("PfTileRotation<D>::rotate", barrier)]))
    assert read <= written_behind and not {r.split(".")[0] for r in read} & written_before, (read, written_before, written_behind)


def test_a_decode_step_that_appends_lets_nobody_start_beside_it():
    """The next step's thread blocks would take the places that its own leave one by one, unevenly over the SMs."""
    src = _source("svlm_decode.cu")
    starts = [line.strip() for line in src.splitlines() if "pdl_launch_dependents" in line]
    assert len(starts) == 2 and all(line.startswith("if (!Append::on)") for line in starts), starts
