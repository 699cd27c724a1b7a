"""Kernels launched while their predecessor still runs keep the rules of lime_common.cuh: no thread leaves ahead of the wait for the
predecessor, and the link-side kernels, beside which a history update runs, signal their dependents behind that wait."""
import ctypes
import glob
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_18239_b200", "csrc")
LINK_SIDE = {"k_link_mlp_tc", "k_link_mlp_d256_tc", "k_link_side_d128", "k_link_side_d256"}


def _code(path):
    text = open(path).read()
    return re.sub(r'//[^\n]*|"(?:[^"\\\n]|\\.)*"', "", text)


def _body(text, at):
    """The braced block that opens at or after `at`."""
    start = text.index("{", at)
    depth = 0
    for i in range(start, len(text)):
        depth += (text[i] == "{") - (text[i] == "}")
        if depth == 0:
            return text[start:i + 1]
    raise AssertionError("unbalanced braces")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = _code(path)
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", text):
            yield m.group(1), _body(text, text.index(")", m.end()))


def _events(body):
    """(what, has this scope or one around it waited) of every wait, signal and exit, in order of the source.  A block of a lambda is a scope
    of its own whose exits are not the kernel's."""
    waited, lambdas = [False], [False]
    for m in re.finditer(r"\{|\}|if \([^;{}]*\) pdl_wait\(\);|pdl_wait\(\);|pdl_launch_dependents\(\);|return;", body):
        t = m.group(0)
        if t == "{":
            waited.append(waited[-1])
            head = body[:m.start()].rstrip()
            lambdas.append(lambdas[-1] or bool(re.search(r"\[&?\]\s*(\([^()]*\)\s*)?(->\s*\w+\s*)?$", head)))
        elif t == "}":
            waited.pop()
            lambdas.pop()
        elif t == "pdl_wait();":
            waited[-1] = True
        elif t == "return;" and not lambdas[-1]:
            yield "exit", waited[-1]
        elif t == "pdl_launch_dependents();":
            yield "signal", waited[-1]


def test_no_kernel_is_left_ahead_of_its_wait():
    with_wait = {name: body for name, body in _kernels() if "pdl_wait();" in body}
    assert LINK_SIDE <= set(with_wait) and len(with_wait) >= 20
    wrong = [name for name, body in with_wait.items() if any(e == ("exit", False) for e in _events(body))]
    assert not wrong, wrong


def test_link_side_kernels_signal_behind_their_wait():
    seen = {}
    for name, body in _kernels():
        if name in LINK_SIDE:
            seen[name] = [w for what, w in _events(body) if what == "signal"]
    assert set(seen) == LINK_SIDE and all(s and all(s) for s in seen.values()), seen


def test_the_update_follows_a_link_side_kernel():
    """Whatever the branch, the launch right before a history update is one of the link side."""
    text = _code(os.path.join(CSRC, "lime_api.cu"))
    body = _body(text, text.index(")", text.index("static lime_status tc_layer_core(")))
    before = body[:body.index("launch_hist_update")]
    launches = re.findall(r"\blaunch_\w+(?=\()", before[before.index("launch_link_attn_tc"):])
    assert launches == ["launch_link_attn_tc", "launch_link_side_d256", "launch_link_side_d128", "launch_link_attn_merge_norm", "launch_link_mlp_tc"]


def test_the_scan_tells_an_exit_ahead_of_the_wait():
    """The scanner itself, on the forms that occur."""
    early = "{ if (bad) { if (x) y(); return; } pdl_launch_dependents(); pdl_wait(); }"
    late = "{ if (bad) { pdl_wait(); return; } auto f = [&](int i) { if (i) return; g(i); }; pdl_wait(); pdl_launch_dependents(); if (b) return; }"
    some = "{ if (!early) pdl_wait(); return; }"
    assert list(_events(early)) == [("exit", False), ("signal", False)]
    assert list(_events(late)) == [("exit", True), ("signal", True), ("exit", True)]
    assert list(_events(some)) == [("exit", False)]


@pytest.fixture(scope="module")
def first_tile(tmp_path_factory):
    """early_first_tile of lime_common.cuh, compiled for the host as it stands there."""
    at = tmp_path_factory.mktemp("split")
    text = open(os.path.join(CSRC, "lime_common.cuh")).read()
    name = "int early_first_tile(int cta, int grid, int n, int late, int late_by)"
    (at / "split.cpp").write_text('#include <cstdint>\nextern "C" ' + name + " " + _body(text, text.index(name)))
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", str(at / "split.cpp"), "-o", str(at / "split.so")], check=True)
    return ctypes.CDLL(str(at / "split.so")).early_first_tile


def test_the_split_of_an_update_beside_the_link_side(first_tile):
    """Every tile belongs to one block, whatever the grid, the late blocks and the tiles; late blocks get `late_by` tiles fewer where there
    are enough, and nothing where the early ones are through before they start."""
    for grid in (1, 2, 37, 147, 148):
        for late in {0, 1, grid // 2, grid - 1, grid}:
            for late_by in (2, 4):
                for n in (0, 1, grid - 1, grid, 3 * grid + 1, 20 * grid + 5):
                    first = [first_tile(c, grid, n, late, late_by) for c in range(grid + 1)]
                    tiles = [b - a for a, b in zip(first, first[1:])]
                    assert first[0] == 0 and first[-1] == n and min(tiles) >= 0, (grid, late, late_by, n)
                    early, behind = tiles[:grid - late], tiles[grid - late:]
                    if early and behind:
                        assert max(behind) <= max(max(early) - late_by + 1, 0), (grid, late, late_by, n, tiles)
                        assert max(early) - min(early) <= 1 and max(behind) - min(behind) <= 1
