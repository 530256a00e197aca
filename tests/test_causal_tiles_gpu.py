"""Causal ELSAA over the bucket tiles and the operand buffer of the chunk
kernels: every table count they are compiled for (one or two 128-bucket
tiles, half a tile), both head dimensions, level blocks below and above a
tile, and outputs that are 16- but not 32-byte aligned. The fp32 output and
log d within 2e-2 of the oracle, D_lr within 1e-2 of itself, as in the other
causal tests; the bf16 output is the fp32 output's rounding, bit for bit."""
import numpy as np
import pytest
import torch

from oracle import causal as orc_causal
from oracle import oracle as orc
from paper_2607_20214_gb300 import build, elsaa
from paper_2607_20214_gb300.workloads import Workload, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_h,L,b,N,base,shift", [
    (64, 4, 32, 512, 256, 16), (64, 8, 64, 1024, 256, 0),
    (64, 16, 128, 1024, 512, 16), (64, 16, 256, 1024, 512, 0),
    (128, 4, 64, 512, 256, 0), (128, 8, 128, 1024, 256, 16),
    (128, 16, 32, 1024, 256, 0), (128, 16, 256, 2048, 512, 16),
    (128, 16, 128, 256, 128, 0),
])
def test_chunks_and_levels(d_h, L, b, N, base, shift):
    build.build()
    wl = Workload("causal tiles", B=1, H=3, N=N, d_h=d_h, dtype="bf16",
                  block=b, race_tables=L, temperature=2.0, seed=95,
                  plane_seed=1095, causal=1, causal_base_len=base)
    x = make_inputs(wl)
    xd = {n: t.cuda() for n, t in x.items()}
    out = []
    for dt in (torch.bfloat16, torch.float32):
        p = elsaa.params_for(wl, out_fp32=int(dt == torch.float32))
        n, pad = x["q"].numel(), shift // dt.itemsize
        buf = torch.full((n + 64,), float("nan"), dtype=dt, device="cuda")
        ls = torch.full((1, 3, N), float("nan"), device="cuda")
        dl = torch.full((1, 3, N), float("nan"), device="cuda")
        ws = elsaa.new_workspace(p, torch.device("cuda:0"))
        ws.fill_(0xFF)  # NaN wherever a state or a row is left out
        elsaa.elsaa_forward(p, xd["q"], xd["k"], xd["v"], xd["w_sort"],
                            xd["w_race"],
                            o=buf[pad:pad + n].view(x["q"].shape),
                            log_d_sparse=ls, d_lr=dl, workspace=ws)
        elsaa.elsaa_check_status(ws)
        assert torch.isnan(buf[:pad]).all()
        assert torch.isnan(buf[pad + n:]).all()
        out.append(buf[pad:pad + n].view(x["q"].shape))
    assert torch.equal(out[0], out[1].bfloat16())
    o = out[1].cpu().numpy()
    pr = dict(orc.params_from_workload(wl), causal_chunk=wl.causal_chunk,
              causal_base_len=wl.causal_base_len)
    for (bi, h), r in orc_causal.forward(x, pr).items():
        assert np.abs(o[bi, h] - r["O"]).max() <= 2e-2, h
        assert np.abs(ls[bi, h].cpu().numpy() -
                      r["log_d_sparse"]).max() <= 2e-2, h
        e = np.abs(dl[bi, h].cpu().numpy() - r["d_lr"]) / r["d_lr"]
        assert e.max() <= 1e-2, h
