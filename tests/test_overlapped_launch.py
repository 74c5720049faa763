"""Kernels that are resident while the kernel before them still writes.

A kernel that calls after_previous() overlaps the one before it, so what the earlier
kernels of its chain write is no constant of its run: a load through ``__ldg``, inline
``ld.global.nc`` or a ``const __restrict__`` pointer may return what was there before,
and may be moved above the wait. This reads the sources: every such kernel, and every
function of its file that it calls, takes the read-only path only for what is complete
before the chain.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1702_01530_gb300", "csrc")

# by file: functions that take the read-only path, for data complete before the chain
COMPLETE = {"lbvh.cu": {"raw": "p"},                  # raw records, from the second kernel on
            "trace.cu": {"k_render": "a.sc.lights"}}  # a scene's lights


def _functions(path):
    """name -> (text from its return type on, body) of the file's function definitions."""
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
    out = {}
    for m in re.finditer(r"\b(\w+)\s*\(", text):
        depth, i = 0, m.end() - 1
        while i < len(text):
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
            if depth == 0:
                break
        tail = re.match(r"\s*\{", text[i:])
        if not tail or m.group(1) in ("if", "for", "while", "switch", "__launch_bounds__"):
            continue
        depth, j = 0, i + tail.end() - 1
        while j < len(text):
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
            if depth == 0:
                break
        out.setdefault(m.group(1), []).append((text[m.start():i], text[i:j]))
    return out


def _overlapped():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        funcs = _functions(path)
        calls = {f: {c for _, body in defs for c in re.findall(r"\b(\w+)\s*(?:<[^;(){}]*>)?\s*\(", body)} & set(funcs)
                 for f, defs in funcs.items()}
        for name in funcs:
            if not name.startswith("k_"):
                continue
            reach, todo = set(), [name]
            while todo:
                f = todo.pop()
                if f not in reach:
                    reach.add(f)
                    todo += calls[f]
            if any("after_previous()" in body for f in reach for _, body in funcs[f]):
                yield os.path.basename(path), name, {f: funcs[f] for f in reach}


KERNELS = list(_overlapped())


def test_the_chains_are_found():
    names = {name for _, name, _ in KERNELS}
    assert {"k_render", "k_resolve", "k_resolve4", "k_tree", "k_tree_up", "k_leaves", "k_top_bins", "k_sah_mid",
            "k_render_nodes", "k_net_fused", "k_bwd_fused", "k_wgrad", "k_update"} <= names


@pytest.mark.parametrize("file,kernel,funcs", KERNELS, ids=[k for _, k, _ in KERNELS])
def test_no_read_only_loads_of_what_the_chain_writes(file, kernel, funcs):
    for name, defs in funcs.items():
        for head, body in defs:
            assert "__restrict__" not in head + body, (kernel, name)
            assert "global.nc" not in body, (kernel, name)
            for arg in re.findall(r"__ldg\(\s*([\w.]+)", body):
                assert COMPLETE.get(file, {}).get(name) == arg, (kernel, name, arg)
