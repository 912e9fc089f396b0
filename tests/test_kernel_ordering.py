"""Ordering rules that the kernels have to keep whatever the hardware happens to do, read off the
sources (breaking one is not something a GPU may be made to show)."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2005_03426_gb300", "csrc")


def _source(name):
    """The file without its comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def _block(text, at):
    """The brace-delimited block that opens at or after position `at`."""
    i = text.index("{", at)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
    raise ValueError("unbalanced braces")


def _kernels(name):
    text = _source(name)
    for m in re.finditer(r"__global__\s+void(?:\s+__launch_bounds__\((?:[^()]|\([^()]*\))*\))?\s*(\w+)\s*\(", text):
        body = _block(text, m.end())
        yield m.group(1), text[m.end():text.index(body, m.end())], body


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")))
def test_cluster_has_started_before_a_partner_is_addressed(name):
    """A CTA may access a partner's shared memory only once the whole cluster is running: the first
    cluster-wide barrier comes before the first access."""
    for kernel, _, body in _kernels(name):
        first = min((body.index(w) for w in ("map_shared_rank", "key_load(", "flag_load(") if w in body), default=None)
        if first is not None:
            assert "cluster.sync()" in body[:first], kernel


def test_a_warp_loads_after_its_lanes_acquire():
    """Where one lane polls a progress key for its warp, a warp barrier follows the poll: the lanes'
    loads are ordered after the acquire by it alone (a shuffle orders no memory)."""
    text = _source("k_sbr.cu")
    at = text.index("auto wait_for")
    body = _block(text, text.index(")", at))
    assert "key_load(" in body and "__syncwarp()" in body[body.index("key_load("):]
    assert text.count("key_load(") == 2  # its definition and this poll


def test_programmatically_serialised_kernels_assume_no_constant_inputs():
    """A kernel that may start before its predecessor has finished (griddepcontrol.wait) runs while its
    inputs are written: none of its pointers is __restrict__, which promises the compiler that they do
    not change and permits read-only loads."""
    found = [(k, args) for k, args, body in _kernels("k_hetrd_large.cu") if "lg_wait()" in body]
    assert len(found) == 6
    for kernel, args in found:
        assert "__restrict__" not in args, kernel
