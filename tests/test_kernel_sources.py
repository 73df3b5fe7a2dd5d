"""Rules that the CUDA sources keep and that no run on a GPU would show broken:
they are read as text."""
from __future__ import annotations

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_15451_gb300", "csrc")


def sources():
    """File name -> text without comments."""
    out = {}
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh", ".h")):
            with open(os.path.join(CSRC, f)) as fh:
                out[f] = re.sub(r"//[^\n]*|/\*.*?\*/", "", fh.read(), flags=re.S)
    return out


def body(text, start):
    """The braces that open after `start`, with what they hold."""
    a = text.index("{", start)
    depth = 0
    for k in range(a, len(text)):
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[a:k + 1]
    raise ValueError("unbalanced braces")


def test_flush_of_a_warp_table_is_decided_by_the_whole_warp():
    """wt_flush holds full-warp collectives.  Whether it runs is voted on by all lanes,
    each with a fill count that it read before any of them went on to add a key, and
    nothing else tests the count."""
    src = sources()
    room = body(src["common.cuh"], src["common.cuh"].index("void wt_make_room("))
    assert re.fullmatch(r"\{\s*int filled = \*\(volatile int32_t \*\)&T\.count;\s*"
                        r"if \(__any_sync\(LD_FULL, filled > WT_LIMIT\)\) wt_flush\(T, G\);\s*\}", room), room
    for f, text in src.items():
        text = text.replace(room, "")
        assert not re.search(r"\bif\s*\([^;{}]*\)\s*\{?\s*wt_flush\(", text), f
        assert not re.search(r"\bif\s*\([^;{}]*WT_LIMIT", text), f


def test_kernels_launched_early_wait_first():
    """A kernel launched by launch_after may start while the one before it runs: its
    first statement waits, once, or it would race with it (and, as a kernel that
    ends without having waited, so would the one after it)."""
    src = sources()
    text = "\n".join(src.values())
    kernels = {}
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(", text):
        kernels[m.group(1)] = body(text, m.end())
    launched = set()
    for f, t in src.items():
        for m in re.finditer(r"\blaunch_after\(\s*(\w+)", t):
            name = m.group(1)
            if name in kernels:
                launched.add(name)
            elif name != "void":  # a variable: every kernel that it may hold (void: the helper itself)
                held = re.findall(r"auto\s+%s\s*=([^;]*);" % name, t)
                assert held, (f, name)
                names = set(re.findall(r"\bk_\w+", " ".join(held)))
                assert names and names <= set(kernels), (f, name)
                launched |= names
    assert len(launched) > 80
    for name in sorted(launched):
        assert re.match(r"\{\s*ld_after_previous\(\);", kernels[name]), name
        assert kernels[name].count("ld_after_previous()") == 1, name
