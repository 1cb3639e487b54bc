"""A CTA may touch another CTA's shared memory only once the whole cluster is
known to run, which a cluster barrier establishes.  In every kernel of the
library a barrier therefore stands, at the top level of the kernel or of its
loop over the models, before the first dereference of a peer's address
(`map_shared_rank`).  Checked on the source text: a missing barrier is a race
that a passing run does not exclude."""
import glob
import os
import re

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1510_01815_gb300", "csrc")


def _kernels(text):
    """(name, body) of each __global__ function of a source file, comments removed."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__global__\s", text):
        start = text.index("{", m.start())
        depth, i = 1, start + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        head = text[m.end():start]
        yield re.findall(r"(\w+)\s*\(", head)[-1], text[start:i]


def _cases():
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        for name, body in _kernels(open(path).read()):
            if "map_shared_rank" in body:
                out.append(pytest.param(body, id=os.path.basename(path) + ":" + name))
    return out


def test_kernels_found():
    assert len(_cases()) >= 4  # fused, tangent, two velocity-field kernels


@pytest.mark.parametrize("body", _cases())
def test_barrier_before_peer_access(body):
    # an address that is only kept for later (`ptr = cluster.map_shared_rank(..) + ..;`)
    # is no access
    accesses = [m.start() for m in re.finditer(r"cluster\.map_shared_rank", body)
                if not re.search(r"\bptr = $", body[:m.start()])]
    barriers = [m.start() for m in re.finditer(r"cluster\.sync\(\)", body)]
    assert barriers and accesses and min(barriers) < min(accesses)
