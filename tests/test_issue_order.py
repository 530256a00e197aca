"""In the block kernel the scores of a tile's later pass overwrite P of the pass
before, so they must wait for the product that reads it. No run shows a missing
wait there (products of one thread finish in order in practice), so the source
is read: the condition for a later pass names that product's barrier."""
import os
import re

from conftest import ROOT


def test_later_scores_wait_for_the_product_before():
    path = os.path.join(ROOT, "paper_2607_20214_gb300", "csrc", "tc_ws.cu")
    with open(path) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    later = re.findall(r"if \(spass > 0\)(.*?);", text, re.S)
    assert len(later) == 1
    assert "up == us" in later[0]
    assert re.search(r"test\(\s*&bars\.v_empty\[\(us - 1\) % VS\],\s*"
                     r"\(us - 1\) / VS & 1\)", later[0])
