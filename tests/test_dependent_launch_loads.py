"""Kernels that wait for the launch before them (griddepcontrol.wait: dep_wait) are on the SMs
while that launch still writes links and flow exponents: the data is not constant for as long as the
reading kernel is resident, which the read-only path asks for.  Checked in the sources, over every
function that such a kernel reaches: no load through that path (__ldg, or a const __restrict__
pointer, from which a compiler may infer it), and the wait before any load and before the kernel
lets its own successor in."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_09764_gb300", "csrc")
# the gauge field: written by plain launches only, which no kernel overlaps
CONSTANT = {"vp_trace"}


def _functions():
    """name -> (parameters, body) of every device function and kernel; comments are taken out."""
    out = {}
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cuh", ".cu")):
            continue
        text = open(os.path.join(CSRC, f)).read()
        text = re.sub(r"//[^\n]*", "", text)
        for m in re.finditer(r"__(?:global|device)__[^;{]*?\b(\w+)\(([^;{]*)\)\s*\{", text):
            depth, k = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[k], 0)
                k += 1
            # __launch_bounds__ and __align__ look like a name with arguments
            name, args = m.group(1), m.group(2)
            if name.startswith("__"):
                name, args = re.findall(r"(\w+)\(([^()]*)", m.group(0))[-1]
            params, body = out.get(name, ("", ""))
            out[name] = (params + args, body + text[m.end():k])
    return out


FUNCTIONS = _functions()
WAIT = ("dep_wait", "dep_wait_launch")


def _calls(body):
    return {n for n in re.findall(r"\b(\w+)\s*[<(]", body) if n in FUNCTIONS}


def _reached(kernel):
    seen, todo = set(), [kernel]
    while todo:
        n = todo.pop()
        if n in seen or n in CONSTANT or n in ("load_link", "load_vec"):
            continue
        seen.add(n)
        todo += _calls(FUNCTIONS[n][1])
    return seen


KERNELS = sorted(n for n in FUNCTIONS if n.startswith("k_") and _reached(n) & set(WAIT))


def test_the_kernels_are_found():
    assert {"k_subsweep_fused", "k_subsweep_pring", "k_subsweep_all", "k_subsweep_split", "k_subsweep_rows", "k_aus_ring",
            "k_aus_pring", "k_aus_split", "k_ape_ring", "k_ape_all", "k_ape_split", "k_flow_stage_ring",
            "k_flow_split"} <= set(KERNELS)


@pytest.mark.parametrize("kernel", KERNELS)
def test_no_read_only_loads_after_the_wait(kernel):
    for n in sorted(_reached(kernel)):
        params, body = FUNCTIONS[n]
        assert "__ldg(" not in body, n
        assert not re.search(r"\bconst\b[^,;()]*__restrict__", params + ";" + body), n
        for args in re.findall(r"\bload_link<([^>]*)>", body) + re.findall(r"\bload_vec<([^>]*)>", body):
            if args.split(",")[0].strip() == "T" and n == "load_link_raw":
                continue
            assert "kLive" in args, (n, args)


@pytest.mark.parametrize("kernel", KERNELS)
def test_the_wait_comes_first(kernel):
    """In the function that waits, no link is read and no successor let in before it."""
    waiting = [n for n in _reached(kernel) if re.search(r"\bdep_wait(_launch)?\(\)", FUNCTIONS[n][1]) and n not in WAIT]
    assert waiting
    for n in waiting:
        before = re.split(r"\bdep_wait(?:_launch)?\(\)", FUNCTIONS[n][1])[0]
        for name in ("load_link", "staple_sum", "row_units", "ring_fetch<", "dep_launch()", "fetch(Int"):
            assert name not in before, (n, name)


def test_every_overlapping_launch_waits():
    """Kernels that go through launch_dependent or one of its callers are kernels that wait."""
    listed = set()
    for f in os.listdir(CSRC):
        text = open(os.path.join(CSRC, f)).read()
        listed |= set(re.findall(r"launch_dependent\((k_\w+)", text))
        for block in re.findall(r"static void \(\*const \w+(?:\[\d\])+\)\([^;]*?;[^;]*;?[^;]*launch_(?:ring|all|split)[^;]*;", text):
            listed |= set(re.findall(r"\bk_\w+(?=<)", block))
    assert listed and listed <= set(KERNELS), listed - set(KERNELS)
