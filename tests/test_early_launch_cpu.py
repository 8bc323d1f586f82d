"""The order of waits and tensor-memory allocations in kernels that start early or let the next kernel start (no GPU): an
allocation waits without a limit, so a successor must not be able to hold columns that this grid still needs."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2505_18976_b200" / "csrc"


def _kernels():
    """(file, kernel, its source without comments) of every kernel."""
    for path in sorted(CSRC.glob("*.cu")):
        src = re.sub(r"//[^\n]*", "", path.read_text())
        for part in re.split(r"(?=__global__)", src)[1:]:
            body = part[:part.index("\n}\n")]
            yield path.name, re.search(r"(\w+_kernel)\s*\(", body).group(1), body


def _with_both():
    return [pytest.param(body, id=f"{f}:{name}") for f, name, body in _kernels()
            if "tcgen05.alloc" in body and ("early_wait()" in body or "early_go()" in body)]


def test_some_kernels_are_looked_at():
    assert len(_with_both()) >= 3


@pytest.mark.parametrize("body", _with_both())
def test_tensor_memory_lies_between_the_wait_and_the_successor(body):
    wait, alloc, go = (body.index(x) for x in ("early_wait()", "tcgen05.alloc", "early_go()"))
    assert body.count("early_wait()") == body.count("early_go()") == body.count("tcgen05.alloc") == 1
    assert wait < alloc < go
    assert "__syncthreads()" in body[alloc:go]


def test_kernels_that_wait_later_follow_a_kernel_of_their_own_call():
    """Kernels with a plain griddepcontrol.wait gather and allocate before it: the kernel before them in the stream is their
    set-up kernel, which takes no tensor memory and is launched the ordinary way."""
    late = {f for f, _, body in _kernels() if "griddepcontrol.wait" in body}
    assert late == {"factgrass.cu", "factgrass_persistent.cu", "grass_sjlt_table.cu"}
    for f in late:
        setup = [(name, body) for g, name, body in _kernels() if g == f and "griddepcontrol.launch_dependents" in body]
        assert len(setup) == 1
        name, body = setup[0]
        assert "tcgen05" not in body and name + "<<<" in (CSRC / f).read_text()
