"""Shared memory of the latent decode's main kernel between its barriers (no GPU).

The four tensor-core warps exchange row maxima and row sums through `red` and the
softmax weights through `sm_p`, in Rows::stage (one 64-token tile) and Rows::finish
(a record at the end of a run of tiles).  Warps run free between two barriers, so
what one writes no other may read, or write again for another purpose, in the same
interval.  The order of accesses and barriers is read from the source and run
through sequences of tiles and records as a CTA meets them.
"""
import os
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_18587_gb300", "csrc",
                      "dar_latent.cu")


def _body(text, name):
    at = re.search(r"__device__ __forceinline__ void %s\(" % name, text).end()
    at = text.index("{", text.index(")\n", at))
    depth = 0
    for i in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return re.sub(r"//[^\n]*", "", text[at:i])
    raise AssertionError("no end of " + name)


def _events(body):
    """Barriers ("|"), writes and reads ("w red", "r sm_p", ...) in program order."""
    found = []
    for m in re.finditer(r"consumer_sync\(\)", body):
        found.append((m.start(), "|"))
    for m in re.finditer(r"\bred\[[^;]*?\](\s*=(?!=))?", body):
        found.append((m.start(), ("w" if m.group(1) else "r") + " red"))
    for m in re.finditer(r"reinterpret_cast<uint32_t \*>\(sm_p\b", body):
        found.append((m.start(), "w sm_p"))
    for m in re.finditer(r"ldsm_x4\(swz\(pbase\b", body):
        found.append((m.start(), "r sm_p"))
    return [e for _, e in sorted(found)]


@pytest.fixture(scope="module")
def events():
    with open(SOURCE) as f:
        text = f.read()
    text = text[text.index("struct Rows"):]
    return {name: _events(_body(text, name)) for name in ("stage", "finish")}


def test_source_is_understood(events):
    assert [e for e in events["stage"] if e != "r red"].count("|") == 2
    assert {"w red", "r red", "w sm_p", "r sm_p"} <= set(events["stage"])
    assert {"w red", "r red", "|"} <= set(events["finish"])


@pytest.mark.parametrize("tiles", [(1, 1, 1), (3, 1, 2), (4, 4)])
def test_no_access_meets_another_between_barriers(events, tiles):
    run = []
    for n in tiles:  # records of n tiles each, one after the other in a CTA's run of work
        for part in ["stage"] * n + ["finish"]:
            run += [e if e == "|" else e + " in " + part for e in events[part]]
    interval = set()
    for e in run + ["|"]:
        if e != "|":
            interval.add(e)
            continue
        for array in ("red", "sm_p"):
            writes = {x for x in interval if x.startswith("w " + array)}
            reads = {x for x in interval if x.startswith("r " + array)}
            assert not (writes and reads) and len(writes) <= 1, sorted(interval)
        interval = set()
