"""Bounded waits of whole warps (csrc/m2l_tc.cu): a wait may run out for some lanes of a warp alone. A lane that left its
role then would keep the others in the role's next warp-wide instruction for ever, which no run may try, so it
is read from the source: lanes leave by a vote between the wait and that instruction, or not at all."""
import os
import re

import pytest

from paper_2006_03515_gb300 import build


def _role(name):
    text = open(os.path.join(build.CSRC, "m2l_tc.cu")).read()
    parts = re.split(r"// -{16} (.*?) -{16}", text)
    body = [parts[k + 1] for k in range(1, len(parts), 2) if parts[k].startswith(name)]
    assert len(body) == 1
    code = re.sub(r"//.*", "", body[0])
    return code[:code.index("__syncthreads()")] if "__syncthreads()" in code else code


def test_the_epilogue_votes_after_its_waits():
    events = re.findall(r"mbar_wait|__all_sync|__syncwarp|tmem_ld\d+|sync\.aligned", _role("epilogue"))
    assert "mbar_wait" in events and "__syncwarp" in events
    waited = False
    for e in events + events:   # (the role is a loop)
        if e == "mbar_wait":
            waited = True
        elif e == "__all_sync":
            waited = False
        else:
            assert not waited, e


@pytest.mark.parametrize("name,head", [("producers", "for (int n = 0; n < total; ++n) {"),
                                       ("index warp", "for (int g = g0; g < g1; g += TC_GRP) {")])
def test_the_others_stay_to_the_last_slot(name, head):   # (the MMA warp waits with one lane)
    code = _role(name)
    loop = code[code.index(head):]
    upto = loop[:loop.rindex("__syncwarp")].replace("if (g + q >= g1) break;", "")   # (the same for all lanes)
    assert "mbar_wait" in upto and not re.search(r"\b(break|return|continue|goto)\b", upto)
    # after it, the producers leave only the loop over the slot's stages early
    assert re.findall(r"for \(int kc|break|return|goto", loop[loop.rindex("__syncwarp"):]) in ([], ["for (int kc", "break"])
