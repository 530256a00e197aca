"""Candidate blocks of the top-k selector on both sides of the rule for query
blocks per CTA (two up to 128 blocks a head and 512 in all, eight beyond), with
block counts that neither divides: exactly the oracle's key sets."""
import pytest

from test_topk_tc_gpu import check, workload
from paper_2607_20214_gb300.workloads import make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,T,c", [(1, 127, 3), (1, 129, 3), (4, 128, 2),
                                   (9, 57, 4), (1, 131, 16)])
def test_key_sets(H, T, c):
    wl = workload(H=H, N=32 * T, block=32, topk_blocks=c, topk=20)
    check(wl, make_inputs(wl))
