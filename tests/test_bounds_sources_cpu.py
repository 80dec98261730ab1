"""The index-checking build covers the kernels that solves, drifts and the preconditioner run in: their vectors and
shared tiles are reached through accessors that check, and every unit that checks reports its error word. Read from
the sources, since a clean run records nothing either way."""

import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2204_14241_gb300", "csrc")


def code(name):
    with open(os.path.join(SRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def body(text, head):
    i = text.index("{", re.search(head, text).end())
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError("unbalanced braces")


def test_accessors_check():
    common, team = code("common.cuh"), code("team.cu")
    for name in ("in_range", "tile_at"):
        assert "HMC_IN(" in body(common, rf"\b{name}\(")
    for name in ("ld_it", "st_it", "d_spin"):
        assert "HMC_IN(" in body(team, rf"\b{name}\(")
    for name in ("ld_field", "out_at", "spec_at"):
        assert "in_range(" in body(code("metric.cu"), rf"\b{name}\(")
    assert "in_range(" in body(code("precond.cu"), r"\bentry\(")


def test_tiles_are_reached_through_the_accessor():
    for name in ("team.cu", "metric.cu", "precond.cu"):
        kernels = code(name).split("bounds_take_tu()")[0]
        assert not re.findall(r"\b(?:tile|rows|half)\[", kernels), name
    assert not re.search(r"\bbase\[", body(code("dft_smem.cuh"), r"\bdft_pass\("))


def test_every_checking_unit_reports():
    status = body(code("hmc.cu"), r"\bhmc_bounds_status\(")
    for name in sorted(os.listdir(SRC)):
        if name.endswith(".cu") and re.search(r"HMC_IN\(|in_range\(|tile_at\(|dft_forward\(", code(name)):
            assert f"bounds_take_{name[:-3]}()" in status, name
