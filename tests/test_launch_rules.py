"""Rules of the kernels' launches that no run on one idle GPU can show broken,
checked in the sources."""

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2109_10687_gb300", "csrc")
FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def _code(path):
    text = open(path).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _functions(code):
    """(head, body) of every device function and kernel."""
    for m in re.finditer(r"__(?:global|device)__[^;{]*\{", code):
        depth, i = 1, m.end()
        while depth and i < len(code):
            depth += {"{": 1, "}": -1}.get(code[i], 0)
            i += 1
        yield m.group(0), code[m.end():i]


WAIT = re.compile(r"pdl_wait\(\)|griddepcontrol\.wait")
TRIGGER = re.compile(r"pdl_trigger\(\)|griddepcontrol\.launch_dependents")
FLAG = re.compile(r"loop_idle\(|\bskip\s*&&")


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_flags_of_the_loop_are_read_where_they_are_visible(path):
    """A kernel that may start before its predecessor has finished reads the
    loop's flags after its wait, or through pdl_enter, which waits in a
    sequence's first launch.  The cluster kernel's first launch is a plain one."""
    for head, body in _functions(_code(path)):
        if "pdl_enter" in head or "sap_cluster_kernel" in head:
            continue
        if not (WAIT.search(body) or TRIGGER.search(body)):
            continue  # never launched early
        for m in FLAG.finditer(body):
            assert WAIT.search(body, 0, m.start()), head


def test_the_first_launch_of_the_cluster_kernel_is_a_plain_one():
    code = _code(os.path.join(CSRC, "sap_cluster.cu"))
    assert re.search(r"numAttrs = with_halo && \(r > 0 \|\| sweep > 0 \|\| colour > 0\) \? 2 : 1;", code)


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_no_block_barrier_under_a_choice_per_warp(path):
    """What runs under sp_switch differs between the warps of a block: no
    function called there, nor the lambda itself, holds a block barrier."""
    code = _code(path)
    bodies = {}
    for head, body in _functions(code):
        name = re.findall(r"(\w+)\s*\(", head)
        if name:
            bodies.setdefault(name[-1] if "__launch_bounds__" in head else name[0], []).append(body)
    for m in re.finditer(r"sp_switch\(\w+, \[&\]\(auto k\) \{", code):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(code[i], 0)
            i += 1
        todo, seen = [code[m.end():i]], set()
        while todo:
            body = todo.pop()
            assert "__syncthreads" not in body and "cl.sync" not in body, body
            for callee in set(re.findall(r"\b(\w+)(?:<[^;{}]*?>)?\(", body)) & set(bodies) - seen:
                seen.add(callee)
                todo += bodies[callee]


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_device_settings_are_not_kept_per_process(path):
    """A kernel's shared-memory limit and a device's properties belong to the
    current device: no function-local static sets or holds them."""
    for m in re.finditer(r"static (?:const )?\w+ \w+ = \[[^\]]*\][^{]*\{(.*?)\}\(\);", _code(path), flags=re.S):
        assert not re.search(r"cudaFuncSetAttribute|cudaDeviceGetAttribute|cudaGetDevice", m.group(1)), m.group(0)
