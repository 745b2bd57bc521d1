"""Kernels launched with programmatic dependent launch are resident while the
kernels before them still write, so nothing they read may go through the
non-coherent path (ld.global.nc: __ldg, const __restrict__ pointers), which is
defined only for memory that stays constant while the kernel runs.  Checked on
the sources: every kernel that launch() starts, and every function it calls."""
import glob
import os
import re

from tests.conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2412_04459_gb300", "csrc")


def _functions():
    """name -> source texts (signature and body) of the device functions."""
    found = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__(?:device|global)__[^;{}]*?\b(\w+)\s*\(", text):
            start = text.find("{", m.end())
            end = text.find(";", m.end())
            if start < 0 or 0 <= end < start:
                continue   # a declaration
            if m.group(1) in ("__launch_bounds__", "__cluster_dims__"):
                name = re.search(r"\b(k_\w+)\s*\(", text[m.start():start]).group(1)
            else:
                name = m.group(1)
            depth, i = 0, start
            while True:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
                if depth == 0:
                    break
            found.setdefault(name, []).append(text[m.start():i])
    return found


def test_overlapped_kernels_load_coherently():
    functions = _functions()
    launched = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        for args in re.findall(r"\blaunch\(([^;]*)", open(path).read()):
            launched |= set(re.findall(r"\bk_\w+", args.split("dim3")[0]))
    waiting = {n for n, bodies in functions.items() if any("begin_kernel();" in b for b in bodies)}
    assert launched == waiting and {"k_preprocess", "k_block_lists", "k_render_fwd"} <= launched
    todo, seen = list(launched), set()
    while todo:
        name = todo.pop()
        if name in seen:
            continue
        seen.add(name)
        for body in functions[name]:
            for bad in ("__ldg", "ld.global.nc", "__restrict__"):
                assert bad not in body, (name, bad)
            todo += [c for c in re.findall(r"\b(\w+)\s*(?:<[^;(){}]*>)?\s*\(", body) if c in functions]
    assert {"fetch_vi", "fwd_walk", "block_lists_entry", "gather_density", "load_sh"} <= seen
