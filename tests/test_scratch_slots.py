"""Scratch slots of a context (csrc/common.cuh) against the functions that hold
them: a slot that grows is freed and allocated anew, so a slot fetched by an
inner solve must not be one that a caller of that solve keeps a pointer to.
Read from the sources; no GPU needed."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1911_04382_gb300", "csrc")
# fetched, used and dropped inside one helper; no caller holds them
TRANSIENT = re.compile(r"SCR_(SCAN2?|TMP\d|EU_\w)$")


def _slots(text):
    return {s for s in re.findall(r"scr<[^>]+>\((SCR_\w+)", text) if not TRANSIENT.match(s)}


def _read(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


# the callers of s_solve: embedding, estimates and densification, single and batched
@pytest.mark.parametrize("caller", ["api.cu", "batch.cu", "filter.cu", "blk.cu"])
def test_inner_solves_use_slots_of_their_own(caller):
    krylov = _read("krylov.cu")
    inner = _slots(_read("core.cu")) | _slots(krylov[:krylov.index("struct PCGArgs")])
    assert inner and not inner & _slots(_read(caller))
