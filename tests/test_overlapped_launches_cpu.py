"""Rules of the kernels that are launched before their predecessor ends (programmatic dependent
launch), checked on their source: what the predecessor writes must not be read through the
non-coherent path, which the dependency wait does not order.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_00253_gb300", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def kernels(text):
    """(name, body) of every __global__ function, comments removed."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__global__", text):
        name = re.search(r"\b(k_\w+)\s*\(", text[m.start():])
        at = text.index("{", m.start() + name.end())
        depth, end = 0, at
        while True:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
            if depth == 0:
                break
        yield name.group(1), text[at:end]


OVERLAPPED = [(f, name, body) for f in FILES for name, body in kernels(open(os.path.join(CSRC, f)).read())
              if "grid_dependency_wait()" in body]


def test_the_overlapped_kernels_are_found():
    assert {name for _, name, _ in OVERLAPPED} == {"k_tile_mm", "k_tpcg_update", "k_tpcg_scalars", "k_tpcg_direction"}


@pytest.mark.parametrize("file,name,body", OVERLAPPED, ids=[k[1] for k in OVERLAPPED])
def test_no_non_coherent_read_of_what_the_predecessor_writes(file, name, body):
    assert not re.search(r"__ldg\s*\(|\.nc\b", body), (file, name)
    # settled data only: the Ritz vectors (made before the loop) and S r (two launches back)
    for arg in re.findall(r"ld_settled\(([^;]*);", body):
        assert "col)" in arg or arg.startswith("u + "), (name, arg)


@pytest.mark.parametrize("file,name,body", OVERLAPPED, ids=[k[1] for k in OVERLAPPED])
def test_the_wait_comes_before_any_read(file, name, body):
    before = body[:body.index("grid_dependency_wait()")]
    assert "->" not in before and "[" not in re.sub(r"extern __shared__[^;]*;|__shared__[^;]*;|smem_raw[^;]*;", "",
                                                    before).replace("dyn4[]", ""), (name, before)
