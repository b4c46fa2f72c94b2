"""Rules of the kernels' source that no run can show (the library is not loaded)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2109_00214_gb300", "csrc")
# device functions of the sources in which the threads of a block meet
MEETING = ("__syncthreads", "species_rates(", "radix_table<true>", "block_exclusive_scan(", "block_faulted(")


def _text(path):
    with open(path, encoding="utf-8") as f:
        s = f.read()
    return re.sub(r"//[^\n]*", "", s)


def _kernels():
    """(name, body) of every kernel."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        s = _text(path)
        for m in re.finditer(r"__global__[^{;]*?\b(k_\w+)\s*\(", s):
            i = s.index("{", m.end())
            depth, j = 0, i
            while True:
                depth += {"{": 1, "}": -1}.get(s[j], 0)
                j += 1
                if depth == 0:
                    break
            out.append((os.path.basename(path) + ":" + m.group(1), s[i:j]))
    return out


KERNELS = dict(_kernels())


def test_the_kernels_are_found():
    assert len(KERNELS) > 40
    assert "__syncthreads" in KERNELS["pd_collide.cu:k_collide"]
    assert "s_runs" in KERNELS["pd_stream.cu:k_push_rz"]


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_blocks_that_meet_stop_together(name):
    """A kernel whose blocks meet at a barrier asks for the fault flag once for
    the whole block: another block may raise it between two warps' reads, and a
    block without some of its warps would go on with shared memory (claim tables,
    run constants, counts) that these were to fill."""
    body = KERNELS[name]
    if any(m in body for m in MEETING):
        assert not re.search(r"st->error\b", body), name
