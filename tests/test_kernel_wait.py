"""Every kernel launched as a programmatic dependent takes its block index from
begin_kernel(), the wait for its predecessor, before anything else, and uses it:
an address that does not depend on it may be loaded before the wait, when the
predecessor's results are not there yet.  Read from the sources, no GPU."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1410_0010_gb300", "csrc")


def _sources():
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        src = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
        out[os.path.basename(path)] = re.sub(r"//[^\n]*", "", src)
    return out


def _kernels(src):
    """(name, body) of every __global__ function."""
    for m in re.finditer(r"__global__ void\s+(?:__launch_bounds__\([^{;]*?\)\s+)?(k_\w+)\(", src):
        start = src.index("{", m.end())
        depth, i = 1, start + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(src[i], 0)
            i += 1
        yield m.group(1), src[start + 1:i - 1]


BODIES = {name: body for src in _sources().values() for name, body in _kernels(src)}
# launched by name, returned by a chooser, or listed by a way of their own (k_deposit<kRows>)
LAUNCHED = sorted({m for src in _sources().values() for pattern in (r"(?:launch_kernel\(|return )(k_\w+)[<,]",
                                                                    r"\b(k_\w+)<k[A-Z]\w*>")
                   for m in re.findall(pattern, src)})


def test_the_launched_kernels_are_found():
    assert len(LAUNCHED) >= 18 and not set(LAUNCHED) - set(BODIES)


@pytest.mark.parametrize("name", LAUNCHED)
def test_block_index_comes_from_the_wait(name):
    first, rest = BODIES[name].strip().split(";", 1)
    assert first.split() == ["const", "unsigned", "block", "=", "begin_kernel()"]
    assert re.search(r"\bblock\b", rest)
    assert "blockIdx" not in rest and "begin_kernel" not in rest
