"""Exact causal attention of the base segments at the edges of its tile
pairs: one tile, an odd last tile, more pairs than CTAs, and keys that grow
along the segment, so that later tiles raise every row's maximum and the
accumulator is rescaled. O (fp32 output) within 2e-2 and log d within 2e-2 of
the oracle, as in the other causal tests."""
import numpy as np
import pytest
import torch

from oracle import causal as orc_causal
from oracle import oracle as orc
from paper_2607_20214_gb300 import build, elsaa
from paper_2607_20214_gb300.workloads import Workload, make_inputs

pytestmark = pytest.mark.gpu


def check(wl, x, heads=None):
    build.build()
    p = elsaa.params_for(wl, out_fp32=1)
    xd = {n: t.cuda() for n, t in x.items()}
    ls = torch.full((wl.B, wl.H, wl.N), float("nan"), device="cuda")
    ws = elsaa.new_workspace(p, torch.device("cuda:0"))
    o = elsaa.elsaa_forward(p, xd["q"], xd["k"], xd["v"], xd["w_sort"],
                            xd["w_race"], log_d_sparse=ls, workspace=ws)
    elsaa.elsaa_check_status(ws)
    pr = dict(orc.params_from_workload(wl), causal_chunk=wl.causal_chunk,
              causal_base_len=wl.causal_base_len)
    for (b, h), r in orc_causal.forward(x, pr, heads=heads).items():
        assert np.abs(o[b, h].cpu().numpy() - r["O"]).max() <= 2e-2, (b, h)
        e = np.abs(ls[b, h].cpu().numpy() - r["log_d_sparse"]).max()
        assert e <= 2e-2, (b, h, e)


def workload(**kw):
    base = dict(name="base", B=1, H=1, N=512, d_h=64, dtype="bf16", block=64,
                race_tables=4, temperature=2.0, seed=81, plane_seed=1081,
                causal=1, causal_base_len=4096)
    base.update(kw)
    return Workload(**base)


@pytest.mark.parametrize("d_h", [64, 128])
@pytest.mark.parametrize("N,base", [(128, 4096), (256, 128), (384, 4096),
                                    (1152, 4096), (2560, 640)])
def test_tile_pairs(d_h, N, base):
    wl = workload(d_h=d_h, N=N, causal_base_len=base)
    check(wl, make_inputs(wl))


@pytest.mark.parametrize("d_h", [64, 128])
def test_more_pairs_than_ctas(d_h):
    wl = workload(d_h=d_h, N=768, causal_base_len=384, B=4, H=60)
    check(wl, make_inputs(wl), heads=[(0, 0), (1, 31), (3, 59)])


@pytest.mark.parametrize("d_h", [64, 128])
def test_rising_maxima(d_h):
    wl = workload(d_h=d_h, N=1280)
    x = make_inputs(wl)
    ramp = torch.linspace(0.1, 6.0, wl.N).view(1, 1, -1, 1)
    x["k"] = (x["k"].float() * ramp).to(torch.bfloat16)
    check(wl, x)
