"""A kernel that lets its successor start early holds its tensor-memory columns by
then: in every kernel that allocates some, a block barrier stands between the
allocation (made by one warp) and the release (by whichever warp comes first).
Without it a successor's CTA on the same SM could take the columns and wait for
a kernel that waits for them.  Checked in the sources: the fault itself would
hang."""

import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2110_01614_gb300" / "csrc"


def unguarded(source):
    """(kernels that both allocate and release, those without the barrier)."""
    code = re.sub(r"//[^\n]*", "", source)
    both, bad = 0, []
    for body in code.split("__global__")[1:]:
        name = re.search(r"(\w+_kernel)\s*\(", body)
        alloc, release = body.find("tcgen05.alloc"), body.find("release_successor()")
        if alloc < 0 or release < 0:
            continue
        both += 1
        if "__syncthreads()" not in body[alloc:release]:
            bad.append(name.group(1) if name else body[:60])
    return both, bad


def test_columns_are_held_before_the_successor_is_released():
    total = 0
    for path in sorted(CSRC.glob("*.cu*")):
        both, bad = unguarded(path.read_text())
        assert not bad, (path.name, bad)
        total += both
    assert total >= 3          # the two width-64 kernels and the Fourier-feature one


def test_the_check_sees_a_missing_barrier():
    text = (CSRC / "query_tc16_w64.cu").read_text()
    code = re.sub(r"//[^\n]*", "", text)
    cut = re.sub(r"__syncthreads\(\);(\s*)wait_for_predecessor", r"\1wait_for_predecessor", code)
    assert cut != code and unguarded(cut)[1] == ["query_w64_small_kernel"]
