"""Order of cluster operations in the kernels' source, checked without a GPU: the
shared memory of another CTA of a cluster may be touched only once that CTA is
known to have started, i.e. after a cluster barrier, and a kernel that arrives at
a cluster barrier waits for it on every way out."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2304_14568_gb300", "csrc")


def _kernels_with_remote_access():
    """(file, kernel, body) of every kernel that addresses another CTA's shared memory."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?(\bk_\w+)\s*\(", src):
            at = src.index("{", m.end())
            depth, end = 1, at + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                end += 1
            body = src[at:end]
            if "map_shared_rank" in body or "mapa" in body:
                out.append((os.path.basename(path), m.group(1), body))
    return out


KERNELS = _kernels_with_remote_access()


def test_the_cg_step_is_among_them():
    assert "k_cg_step" in [k for _, k, _ in KERNELS]


@pytest.mark.parametrize("file,kernel,body", KERNELS, ids=[k for _, k, _ in KERNELS])
def test_no_remote_access_before_a_cluster_barrier(file, kernel, body):
    first = min(body.find(w) for w in ("map_shared_rank", "mapa") if w in body)
    before = body[:first]
    assert "barrier_wait(" in before or ".sync()" in before, f"{file} {kernel}"


@pytest.mark.parametrize("file,kernel,body", KERNELS, ids=[k for _, k, _ in KERNELS])
def test_every_arrival_is_waited_for(file, kernel, body):
    arrive = body.find("barrier_arrive(")
    if arrive < 0:
        return
    at = arrive
    for m in re.finditer(r"\breturn\b", body):
        if m.start() > arrive:
            assert "barrier_wait(" in body[at:m.start()] or "barrier_wait(" in body[arrive:m.start()], f"{file} {kernel}"
