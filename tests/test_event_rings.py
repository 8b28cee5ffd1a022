"""The events of a warp go to a ring in shared memory at places that its lanes
count from a mask.  Lanes that take a branch together need not run it together,
so a mask of the lanes active inside a branch may name some of them only, and
two groups would write to the same places: the masks behind note_event come from
ballots of the whole warp, taken before the branch."""
import re
from pathlib import Path

import paper_2008_10468_gb300

SRC = Path(paper_2008_10468_gb300.__file__).parent / "csrc" / "qed.cu"


def test_ring_places_come_from_whole_warp_ballots():
    text = re.sub(r"//[^\n]*", "", SRC.read_text())
    calls = [m.start() for m in re.finditer(r"\bnote_event\(", text)]
    assert len(calls) >= 4   # the definition, the thread pass, the sampler pass, the lane passes
    for at in calls[1:]:
        # the mask counted in the call, or in the place computed just before it
        near = text[max(0, at - 300):at + 200]
        masks = re.findall(r"__popc\((\w+) & \(\(1u << lane\) - 1u\)\)", near)
        assert masks, near
        for m in masks:
            sets = re.findall(r"\b%s = (\w+)\(([^;]*);" % m, text[:at])
            assert sets, m
            assert sets[-1][0] == "__ballot_sync", (m, sets[-1])
            assert sets[-1][1].startswith(("kAll", "0xffffffffu")), sets[-1]
