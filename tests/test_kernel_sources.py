"""Rules of the device code that no run on a healthy device can show broken (no GPU needed)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_04466_b200", "csrc")


def _code(path):
    """Source without comments."""
    return re.sub(r"/\*.*?\*/|//[^\n]*", "", open(path).read(), flags=re.S)


SOURCES = {os.path.basename(f): _code(f) for f in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))}
ALLOCATING = [n for n, c in SOURCES.items() if "tcgen05.alloc" in c]


@pytest.mark.parametrize("name", ALLOCATING)
def test_dependents_are_released_behind_the_tensor_memory_allocation(name):
    """An allocation of tensor memory waits without a limit.  Once every block of a grid has released its dependents these may become
    resident beside it, so a block that released first could find its columns taken by a block that waits for it in turn: every block
    allocates, meets the others of its block at a barrier, and only then releases."""
    code = SOURCES[name]
    last_alloc, release = code.rindex("tcgen05.alloc"), code.index("pdl_launch_dependents()")
    assert code.count("pdl_launch_dependents()") == 1
    assert last_alloc < release and "__syncthreads()" in code[last_alloc:release]


def test_the_rule_above_looks_at_every_allocating_kernel():
    assert set(ALLOCATING) == {"conv_tc.cu", "conv_first_tc.cu", "conv_first_fused.cu", "conv_s2_tc.cu", "conv_lstm_tc.cu", "post_tc.cu"}
    launched = [n for n in ALLOCATING if re.search(r"tcgen05\.alloc", SOURCES[n]) and SOURCES[n].count("__global__") == 1]
    assert launched == ALLOCATING          # one kernel per file: an order in the file is an order in the kernel


def test_no_warp_vote_takes_whatever_lanes_happen_to_be_active():
    """Nothing guarantees that the lanes __activemask() sees are those that reach the vote behind it together."""
    assert [n for n, c in SOURCES.items() if "__activemask" in c] == []


def test_status_codes_name_the_kernel():
    """Every bounded wait reports a code of its kernel's own hundreds."""
    bases = dict(re.findall(r"(WAIT_[A-Z0-9_]+) = (0x[0-9A-F]+)", SOURCES["tc_ptx.cuh"]))
    values = [int(v, 16) for v in bases.values()]
    assert len(set(v >> 8 for v in values)) == len(values) and all(v & 0xFF == 0 for v in values)
    of_file = {}
    for name in [n for n in SOURCES if n.endswith(".cu") and n not in ("wait_probe.cu", "tt_api.cu")]:
        code = SOURCES[name]
        waits = re.findall(r"mbar_wait(?:_uniform)?\([^;]*?p\.status, ([^,]+), (?:p\.)?wait_limit\)", code) + re.findall(r"atomicCAS\(p\.status, 0, ([^)]+)\)", code)
        assert len(waits) == code.count("mbar_wait(") + code.count("mbar_wait_uniform(") + code.count("atomicCAS(p.status")
        for w in waits:
            m = re.fullmatch(r"(?:tc::)?(WAIT_[A-Z0-9_]+)((?: \+ .*)?)", w)
            assert m and m.group(1) in bases, (name, w)
            of_file.setdefault(m.group(1), {}).setdefault(name, []).append(m.group(2))
        # kernels without an abort flag wait by a limit of their own, which the host gives them too, and report behind the wait
        calls = re.sub(r"bool sw_wait\([^{]*\{", "", code)
        own = re.findall(r"\b(?:mbar_wait_limit|sw_wait)\([^;]*?, (?:p\.)?(\w+)\)[;,)]", calls)
        assert len(own) == calls.count("mbar_wait_limit(") + calls.count("sw_wait(") and set(own) <= {"wait_limit", "PRE_LAND_CYCLES"}
        if own:
            assert "p.wait_limit > 0 ? p.wait_limit :" in code and "atomicCAS(p.status" in code
    for base, files in of_file.items():
        assert len(files) == 1, f"{base} is used by {sorted(files)}"
    assert set(of_file) == set(bases) - {"WAIT_PROBE"}


@pytest.mark.parametrize("name", [n for n, c in SOURCES.items() if "__global__" in c and re.search(r"umma_commit_(both|pair)\(", c)])
def test_producers_of_a_pair_wait_for_their_last_free_signals(name):
    """The commits that free a ring's stages signal barriers in both blocks of a pair.  The second block must still be there when the last of
    them arrive: every producer takes a turn of its ring behind its loop, as if it had something left to load, before the blocks meet."""
    body = SOURCES[name].split("__global__", 1)[1].rsplit("if (PAIR) cluster_sync_all();", 1)[0]
    waits = re.findall(r"mbar_wait\(smem_u32\((\w*empty\w*) \+ stage\), phase \^ 1u", body)
    rings = re.findall(r"commit(?:_pair)?\((\w*empty\w*) \+", body)      # freed by commits ("empty0": the address of empty_bar)
    assert rings and sorted(waits) == sorted(2 * [{"empty0": "empty_bar"}.get(r, r) for r in dict.fromkeys(rings) if r in waits or r == "empty0"])
    tails = re.findall(r"for \([^;]*; PAIR && (\w+) < (\w+) && ok;", body)
    assert len(tails) == len(waits) // 2


@pytest.mark.parametrize("producers,stages", [(2, 10), (2, 5), (1, 2), (3, 4), (3, 8)])
def test_a_turn_of_the_ring_waits_for_each_stages_last_use_once(producers, stages):
    """The index arithmetic of that turn: producer j owns iterations j, j + producers, ...; the wait in front of iteration g is for the use
    `stages` iterations before it.  All producers' turns together wait for the last use of every stage, and for nothing that never comes."""
    for per_unit in (1, 9, 18, 27, 36):
        for units in (0, 1, 2, 5):
            total, waited = per_unit * units, []
            for j in range(producers):
                stage, phase, it = j % stages, 0, j
                g = j
                for _ in range(units):
                    while it < per_unit:
                        assert (stage, phase) == (g % stages, g // stages & 1)
                        it, g, stage = it + producers, g + producers, stage + producers
                        if stage >= stages:
                            stage, phase = stage - stages, phase ^ 1
                    it -= per_unit
                while it < stages:
                    assert (stage, phase) == (g % stages, g // stages & 1)
                    waited.append(g - stages)
                    it, g, stage = it + producers, g + producers, stage + producers
                    if stage >= stages:
                        stage, phase = stage - stages, phase ^ 1
            assert sorted(waited) == list(range(total - stages, total))     # negative: never used, the wait returns at once


def test_every_kernel_that_waits_is_given_the_contexts_limit():
    """A context's ticks pass its limit and its status word to every kernel that has both."""
    lines = [line for line in SOURCES["tt_api.cu"].splitlines() if ".status = ctx->status_dev" in line]
    assert len(lines) == 7
    for line in lines:
        assert re.search(r"(\w+)\.status = ctx->status_dev;.* \1\.wait_limit = ctx->wait_limit;", line), line
