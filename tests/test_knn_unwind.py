"""The epilogue warps of the tensor-core k-NN kernel meet at a named barrier
once per work item, and any warp of the block may raise the abort flag at any
time.  Every epilogue warp must leave its item loop after the same item, or the
others wait at that barrier for ever.  Two parts: the rule by which the source
ends an item, and every interleaving of two warps and the flag under that rule."""
import os
import re

from conftest import ROOT


def _item_end_rule():
    """'common' when the loop's condition comes from a value that the item's last
    barrier gives to all warps, 'own' when a warp reads the flag after it."""
    src = open(os.path.join(ROOT, "paper_1807_08692_gb300", "csrc", "hd_knn.cu")).read()
    body = src[src.index("// ---------------- epilogue: warps 2..9"):]
    body = body[:body.index("tc::fence_before_sync();\n    __syncthreads();")]
    barriers = [m.start() for m in re.finditer(r"bar\.sync 1,|tc::bar_any<1, EPI>", body)]
    assert len(barriers) == 2, "one barrier before the two halves of a row meet, one at the end of the item"
    tail = body[body.rindex("\n", 0, barriers[-1]):]
    statement = tail[:tail.index(";\n")]
    after = tail[tail.index(";\n"):]
    if "abort_flag" in after:
        return "own"
    return "common" if re.search(r"\bok = !tc::bar_any<1, EPI>\(.*abort_flag\)", statement) else "unknown"


def _stuck(rule, items=3):
    """Whether some interleaving ends with one warp waiting for one that has left.
    A warp's state: (item, step); steps 0 read the flag before the barrier (rule
    'common'), 1 at the barrier, 2 read the flag after it (rule 'own'), 3 left."""
    start = ((0, 0, False), (0, 0, False), False)
    seen, todo = {start}, [start]
    while todo:
        a, b, flag = todo.pop()
        nxt = []
        if not flag:
            nxt.append((a, b, True))
        for me, other, swap in ((a, b, False), (b, a, True)):
            item, step, saw = me
            if step == 0:
                new = (item, 1, flag if rule == "common" else False)
            elif step == 2:
                new = (item, 3, saw) if flag or item + 1 == items else (item + 1, 0, False)
            else:
                continue
            nxt.append((other, new, flag) if swap else (new, other, flag))
        if a[1] == b[1] == 1:
            if rule == "common":
                leave = a[2] or b[2] or a[0] + 1 == items
                new = (a[0], 3, False) if leave else (a[0] + 1, 0, False)
            else:
                new = (a[0], 2, False)
            nxt.append((new, new, flag))
        if (a[1] == 1 and b[1] == 3) or (b[1] == 1 and a[1] == 3):
            return True
        for s in nxt:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return False


def test_all_warps_leave_after_the_same_item():
    assert _stuck("own") and not _stuck("common")
    assert _item_end_rule() == "common"
