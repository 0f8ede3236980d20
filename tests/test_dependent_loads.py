"""Kernels that may be resident before the kernels they follow have finished read what those write
by ordinary loads.

A kernel that calls after_previous() can be launched ahead of the end of its predecessors.  The
read-only path (__ldg, const __restrict__ parameters) promises data that nobody writes during the
kernel's life, so it is left to what is complete before the first kernel of a chain: the view
descriptors, the supervision, the upstream gradients and the plane parameters.  The sources are read
as text: a wrong value would need an unlucky order of loads, which no run can be made to show."""
import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2412_03451_gb300", "csrc")
FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))
COMPLETE = re.compile(r"&(?:vw->|views\[|a\.views\[|a\.gt_depth\[|a\.gt_normal\[|a\.dLdD\[|a\.dLdN\[|"
                      r"a\.center\[|a\.quat\[|a\.radii\[)")


def device_functions():
    """name -> (parameters, body) of every kernel and device function."""
    out = {}
    for path in FILES:
        src = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        for m in re.finditer(r"__(?:global|device)__\s", src):
            head = re.compile(r"[^;{}]*?\b([A-Za-z_]\w*)\s*\(((?:[^(){};]|\([^()]*\))*)\)\s*\{").match(src, m.end())
            if not head:
                continue
            depth, i = 1, head.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            out[head.group(1)] = (head.group(2), src[head.end():i])
    return out


FUNCS = device_functions()
EARLY = sorted(n for n, (_, body) in FUNCS.items() if "after_previous()" in body)


def reached(name):
    seen, todo = {name}, [name]
    while todo:
        for callee in re.findall(r"\b([A-Za-z_]\w*)\s*(?:<[^;(){}]*>)?\s*\(", FUNCS[todo.pop()][1]):
            if callee in FUNCS and callee not in seen:
                seen.add(callee)
                todo.append(callee)
    return seen


def test_the_chain_is_found():
    assert {"k_project", "k_scan_sums", "k_scan_apply", "k_pair_scatter", "k_sort", "k_splat", "k_chain",
            "k_chain_adam"} <= set(EARLY)
    assert {"run_strip", "walk_strip", "flush", "run_hard", "tile_setup", "load_state"} <= reached("k_splat")
    assert {"chunk_record_range", "pair_record", "entry_key"} <= reached("k_pair_scatter")


@pytest.mark.parametrize("kernel", EARLY)
def test_no_read_only_loads_of_what_the_chain_writes(kernel):
    for f in sorted(reached(kernel)):
        params, body = FUNCS[f]
        loads = re.findall(r"__ldg\(\s*([^()]*(?:\([^()]*\)[^()]*)*)\)", body)
        assert len(loads) == body.count("__ldg("), f
        assert [x for x in loads if not COMPLETE.match(x)] == [], f
        promised = [p for p in params.split(",") if re.search(r"\bconst\b.*__restrict__", p)]
        assert [p for p in promised if "ps_view" not in p] == [], f
