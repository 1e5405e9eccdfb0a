"""How the sources use the warp-collective tensor-memory instructions, read as
text: the rules that a run cannot show to be kept, since a broken one goes
wrong only where the compiler or the scheduler makes it."""
from __future__ import annotations

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_09184_gb300", "csrc")


def _read(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def _functions(text):
    """{name: body} of the brace-delimited functions (device ones, members included)"""
    out = {}
    for m in re.finditer(r"SFHE_DEV\s+(?:static\s+)?\w+\s+(\w+)\(", text):
        i = text.index("{", m.end())
        depth, j = 1, i + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        out[m.group(1)] = text[i:j]
    return out


def test_collective_instructions_follow_a_warp_barrier():
    """PTX leaves a .sync.aligned instruction undefined in a diverged warp:
    each sequence of them starts with __syncwarp()"""
    fns = _functions(_read("round_mma.cuh"))
    collective = {n for n, body in fns.items() if ".sync.aligned" in body}
    assert {"tmem_alloc", "tmem_dealloc", "tmem_st8", "tmem_ld8", "tmem_wait_st", "tmem_wait_ld"} <= collective
    guarded = set()
    for name, body in fns.items():
        first = min([m.start() for c in collective - {name} for m in re.finditer(r"\b%s\b" % c, body)] +
                    [m.start() for m in re.finditer(r"\.sync\.aligned", body)], default=None)
        if first is not None and "__syncwarp();" in body[:first]:
            guarded.add(name)
    assert {"tmem_alloc", "tmem_dealloc", "store_row", "load_row"} <= guarded
    # the unguarded ones are called from the guarded ones only
    for name in collective - guarded:
        for other, body in fns.items():
            if other != name and re.search(r"\b%s\b" % name, body):
                assert other in guarded, (name, other)
        for f in os.listdir(CSRC):
            if f.endswith((".cu", ".cuh")) and f != "round_mma.cuh":
                assert not re.search(r"\b%s\b" % name, _read(f)), (name, f)


def test_loaded_registers_depend_on_the_wait():
    """the compiler may move a use of a loaded register above a wait that does
    not name it: the wait takes the registers, and every load has one before
    the first use"""
    fns = _functions(_read("round_mma.cuh"))
    wait = fns["tmem_wait_ld"]
    assert re.search(r'asm volatile\("" : "\+r"\(w\[i\]\)\)', wait[wait.index("wait::ld"):])
    body = fns["load_row"]
    loads = [m.end() for m in re.finditer(r"tmem_ld8\(reinterpret_cast<u32\(&\)\[8\]>\(r\[8 \* q\]\), d[^;]*;", body)]
    assert len(loads) == len(re.findall("tmem_ld8", body)) == 2
    for at in loads:
        assert body[at:].lstrip().startswith("tmem_wait_ld(r);")


def test_a_matrix_product_that_runs_out_of_time_is_the_last():
    """stage S: a thread whose wait ran out issues no further product, keeps
    the phase it waited for, and waits once more (bounded) before the kernel
    gives its tensor memory back"""
    text = _read("kernels.cuh")
    i = text.index("auto stage_s_mma")
    body = text[i:text.index("auto stage_s =", i)]
    loop, end = body.split("return alive;")[0].rsplit("sum[(size_t)i * N] = prev[i] + w[i];", 1)
    rows = loop.index("alive = mbar_wait(&row_bar[wg]")
    issue = loop.index("RM::issue")
    guard = loop.index("if (row == 0 && alive)")
    assert rows < guard < issue and loop.count("RM::issue") == 1
    done = loop.index("if (alive) alive = mbar_wait(&mma_bar[wg]")
    assert issue < done < loop.index("if (alive) mma_phase ^= 1u;") < loop.index("RM::load_row")
    assert loop.count("mma_phase ^=") == 1
    assert re.search(r"if \(!alive\) mbar_wait\(&mma_bar\[wg\], mma_phase, SFHE_WAIT_TRIES, SFHE_WAIT_NS\);", end)
