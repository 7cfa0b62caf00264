"""The solver kernels' reduction slots: a sum's partials may be overwritten
only after a grid barrier that follows their last read.  Read from the source:
for every pair of phases that can follow each other without a barrier, the
slots that the first reads after its last barrier and those that the second
writes before its first barrier have to be different ones."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_22215_gb300", "csrc")
SOURCE = open(os.path.join(CSRC, "solve.cu")).read()


def slot_numbers():
    names = {}
    for item in re.search(r"enum Slot \{(.*?)\};", SOURCE, re.S).group(1).split(","):
        name, value = (s.strip() for s in item.split("="))
        names[name] = names[value] if value in names else int(value)
    return names


def body(name):
    at = re.search(r"__device__ [^;{}]*\b%s\([^;{}]*\)\s*\{" % name, SOURCE).end()
    depth, end = 1, at
    while depth:
        depth += {"{": 1, "}": -1}.get(SOURCE[end], 0)
        end += 1
    # refine_residual without its fold step (the restarted form), whose barrier comes first
    return re.sub(r"if \(fold\) \{.*?\n    \}", "", SOURCE[at:end], flags=re.S)


def events(name):
    """(kind, slots) of a phase in source order: "read", "write", "barrier"."""
    slots, out = slot_numbers(), []
    for m in re.finditer(r"grid_reduce_read<(\d)[^>]*>\([^;]*?(SL_\w+)(?: \+ (\d))?[,)]"
                         r"|block_(?:reduce|max)_store<(\d)>\([^;]*?(SL_\w+)(?: \+ (\d))?[,)]"
                         r"|group_sync\(|sweep_levels<", body(name)):
        rn, rs, ro, wn, ws, wo = m.groups()
        if rn:
            out.append(("read", {slots[rs] + int(ro or 0) + k for k in range(int(rn))}))
        elif wn:
            out.append(("write", {slots[ws] + int(wo or 0) + k for k in range(int(wn))}))
        else:
            out.append(("barrier", set()))
    return out


# the initial sums are followed by the diagonal or DIC application, the restarted form's residual, or (a system
# that starts converged) the true residual; the true residual by itself follows whichever sum stopped the loop
PAIRS = [("phase_init", f) for f in ("diag_pass", "dic_apply", "refine_residual", "true_residual")]
PAIRS += [(f, "true_residual") for f in ("diag_pass", "update_pass", "refine_residual", "amul_sigma")]


@pytest.mark.parametrize("first,second", PAIRS)
def test_no_slot_is_rewritten_while_it_may_be_read(first, second):
    read = set()
    for kind, slots in events(first):
        read = set() if kind == "barrier" else read | slots if kind == "read" else read
    written = set()
    for kind, slots in events(second):
        if kind == "barrier":
            break
        written |= slots if kind == "write" else set()
    assert read and written
    assert not read & written
