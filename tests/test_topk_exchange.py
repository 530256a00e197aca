"""The top-k selection's pass for rows with many open candidates: in each turn
two lanes of a warp hand their rows' words over in shared memory and read the
result from the same words, which other lanes write in the next turn. Only a
warp barrier at the end of a turn orders that write behind the read, and no
run shows its absence, so the source is read."""
import os
import re

from conftest import ROOT


def _body(text, start):
    depth = 0
    for i in range(text.index("{", start), len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[text.index("{", start) + 1:i]
    raise AssertionError("unbalanced braces")


def test_a_turn_ends_with_a_warp_barrier():
    path = os.path.join(ROOT, "paper_2607_20214_gb300", "csrc", "topk_tc.cu")
    with open(path) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    turns = [m.start() for m in re.finditer(r"while \(rest\)", text)]
    assert len(turns) == 1
    body = _body(text, turns[0])
    assert "pair_sync();" in body
    assert body.rstrip().endswith("__syncwarp();")
