"""The hard points' search keeps its warps whole: the distance that other warps
lower meanwhile is read by one lane and broadcast before any branch.  Lanes that
each read it could see different values and part in front of a full-warp ballot,
which is undefined.  Checked in the source: the fault itself could hang."""

import pathlib
import re

SOURCE = pathlib.Path(__file__).resolve().parent.parent / "paper_2110_01614_gb300" / "csrc" / "mesh_tree.cu"


def search(text):
    code = re.sub(r"//[^\n]*", "", text)
    body = code[code.index("warp_search("):]
    return body[:body.index("\n}\n")]


def unbroadcast(body):
    """Reads of the shared distance that do not go through lane 0 and a shuffle."""
    bad = []
    for m in re.finditer(r"\*\s*\(volatile unsigned \*\)\s*shared_best", body):
        before = body[:m.start()].rsplit(";", 1)[1]
        target = re.match(r"\s*if \(lane == 0u\) (\w+) = $", before)
        after = body[m.end():]
        if not target or not re.match(
                r";\s*const float (\w+) = __uint_as_float\(__shfl_sync\(0xffffffffu, %s, 0\)\);"
                % target.group(1), after):
            bad.append(body[m.start() - 60:m.end()])
    return bad


def test_the_shared_distance_is_broadcast():
    body = search(SOURCE.read_text())
    uses = len(re.findall(r"\bshared_best\b", body))
    # the parameter, two null tests, the broadcast read and lane 0's atomicMin
    assert uses == 5 and "if (shared_best && lane == 0) atomicMin(shared_best, m);" in body
    assert unbroadcast(body) == []


def test_the_check_sees_a_read_by_every_lane():
    body = search(SOURCE.read_text())
    old = re.sub(r"if \(lane == 0u\) bits = ", "bits = ", body)
    assert old != body and len(unbroadcast(old)) == 1
