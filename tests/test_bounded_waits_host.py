"""Bounded waits in the row passes' source, checked without a GPU: a consumer warp
goes on into full-mask shuffles and warp barriers after a wait, so the outcome of a
wait that can run out must be one for the whole warp (a vote), not each lane's own."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2304_14568_gb300", "csrc")


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def _raw_waits(src):
    """Uses of a lane's own wait outside the definitions and the votes over them."""
    src = re.sub(r"__device__ __forceinline__ bool \w*wait\([^)]*\)\s*\{.*?\n?\}", "", src, flags=re.S)
    return [m.start() for m in re.finditer(r"(?<![\w])(mbar_wait|flag_wait)\(", src)], src


@pytest.mark.parametrize("name", ["rowpriv.cu", "rowpass.cu"])
def test_consumers_take_one_answer_a_warp(name):
    at, src = _raw_waits(_source(name))
    consumers = src.index("int cw = warp - ")       # producers come before
    assert not [a for a in at if a > consumers], name


def test_a_turn_that_never_came_adds_nothing():
    src = _source("rowpriv.cu")
    item = src[src.index("process_item("):src.index("k_rowpass_priv(")]
    wait = item.index("flag_wait(S.turn_a")
    adds = [m.start() for m in re.finditer(r"acc\[[^;]*\]\s*\+?=", item) if m.start() > wait]
    assert adds and re.search(r"if \(!S\.ok\) return;", item[wait:adds[0]])


def test_turns_are_taken_whatever_their_address():
    """0 is a possible address in shared memory: it cannot mean "no turns"."""
    src = _source("rowpriv.cu")
    assert "S.turn_a" in src and not re.search(r"\(\s*S\.turn_a\s*(\)|&&|\|\||[!=]=)|\?[^;]*turns\[[^;]*:", src)
