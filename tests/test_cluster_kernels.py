"""Kernels that store into the shared memory of the other blocks of their cluster: a cluster barrier that every block
passes stands in front of the first such store (a block may not be written to before it has started).  Read from the
source: on the GPU a missing barrier shows only by chance."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_15461_gb300", "csrc")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for body in re.split(r"(?=\n(?:template [^\n]*\n)?__global__ )", src)[1:]:
            end = body.find("\n}\n")
            body = body[:end] if end >= 0 else body
            if "map_shared_rank" in body:
                name = re.search(r"(k_\w+)\s*\(", body).group(1)
                yield pytest.param(body, id=name)


def test_there_is_one():
    assert [p.id for p in _kernels()] == ["k_gemv_reduce"]


@pytest.mark.parametrize("body", list(_kernels()))
def test_blocks_have_started_before_the_first_remote_store(body):
    lam = re.search(r"\n    auto (\w+) = \[&\](?:(?!\n    };).)*map_shared_rank.*?\n    };", body, re.S)
    if lam:   # the store is in a lambda: what counts is its first call
        body = body.replace(lam.group(0), "")
    before = body[:re.search(r"\b" + lam.group(1) + r"\(" if lam else "map_shared_rank", body).start()]
    arrive, wait = before.find("cluster_arrive();"), before.find("cluster_wait();")
    assert 0 <= arrive < wait
    # every thread takes part in both: neither stands in a block of its own
    for pos in (arrive, wait):
        line = before[before.rfind("\n", 0, pos) + 1:pos]
        assert line == "    ", line
    assert "return" not in before[:wait]
