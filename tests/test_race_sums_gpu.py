"""A = Phi_K^T 1 and B = Phi_K^T V come from the same additions: with values
of one, every column of B equals A bit for bit, over chunks of one key tile to
many, ragged ends and every number of bucket tiles. (The additions of the
tensor cores truncate: an A summed otherwise leaves its error in Num / Den.)"""
import pytest
import torch

from paper_2607_20214_gb300 import build, elsaa
from paper_2607_20214_gb300.workloads import Workload, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_h,L,N", [
    (128, 4, 512), (128, 5, 1088), (128, 8, 4800), (128, 12, 8192),
    (128, 16, 65536), (64, 4, 576), (64, 8, 65536), (64, 16, 8192),
])
def test_a_is_b_for_values_of_one(d_h, L, N):
    build.build()
    wl = Workload(name="sums", B=1, H=4, N=N, d_h=d_h, dtype="bf16", block=64,
                  race_tables=L, recipe="plain", temperature=2.0, seed=83,
                  plane_seed=1083)
    dev = torch.device("cuda:0")
    x = {n: t.to(dev) for n, t in make_inputs(wl).items()}
    p = elsaa.params_for(wl)
    ws = elsaa.new_workspace(p, dev)
    elsaa.elsaa_forward(p, x["q"], x["k"], torch.ones_like(x["v"]),
                        x["w_sort"], x["w_race"], workspace=ws)
    A, B = elsaa.elsaa_forward_race_summaries(p, ws)
    elsaa.elsaa_check_status(ws)
    assert A.min() > 0
    assert torch.equal(B.reshape(*A.shape, d_h),
                       A[..., None].expand(*A.shape, d_h))
