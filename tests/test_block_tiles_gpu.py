"""The tensor-core block kernel at the edges of its tiles: fewer tiles than
buffers, CTAs that change heads, half-empty last tiles, key blocks of 32 and
64 inside a 128-query tile, outputs that are 16- but not 32-byte aligned.
Tolerance 2e-2, as for every bf16 output against the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2607_20214_gb300 import build, elsaa
from paper_2607_20214_gb300.workloads import Workload, make_inputs

pytestmark = pytest.mark.gpu


def run(wl, x, shift=0, **over):
    build.build()
    dev = torch.device("cuda:0")
    p = elsaa.params_for(wl, **over)
    xd = {n: t.to(dev) for n, t in x.items()}
    dt = torch.float32 if over.get("out_fp32") else torch.bfloat16
    n = x["q"].numel()
    pad = shift // dt.itemsize
    buf = torch.full((n + 64,), float("nan"), dtype=dt, device=dev)
    o = buf[pad:pad + n].view(x["q"].shape)
    ws = elsaa.new_workspace(p, dev)
    elsaa.elsaa_forward(p, xd["q"], xd["k"], xd["v"], xd["w_sort"],
                        xd["w_race"], o=o, workspace=ws)
    elsaa.elsaa_check_status(ws)
    assert torch.isnan(buf[:pad]).all() and torch.isnan(buf[pad + n:]).all()
    return o.float().cpu().numpy()


def workload(**kw):
    base = dict(name="tiles", B=1, H=2, N=1024, d_h=64, dtype="bf16",
                block=64, race_tables=8, recipe="plain", temperature=2.0,
                seed=61, plane_seed=1061)
    base.update(kw)
    return Workload(**base)


def check(wl, got, x):
    for (b, h), r in orc.forward(x, orc.params_from_workload(wl)).items():
        assert np.abs(got[b, h] - r["O"]).max() <= 2e-2, (wl, b, h)


@pytest.mark.parametrize("d_h,b,N,L", [
    (64, 32, 32, 4), (64, 32, 160, 8), (64, 32, 2080, 16), (64, 64, 64, 8),
    (64, 64, 192, 4), (64, 64, 4800, 8), (64, 128, 128, 8),
    (64, 128, 1920, 16), (128, 32, 352, 16), (128, 64, 64, 16),
    (128, 64, 960, 4), (128, 128, 128, 16), (128, 128, 1280, 8),
    (64, 256, 512, 8), (64, 256, 2304, 16), (128, 256, 1280, 4),
])
def test_tile_edges(d_h, b, N, L):
    wl = workload(d_h=d_h, block=b, N=N, race_tables=L, H=3)
    x = make_inputs(wl)
    check(wl, run(wl, x), x)


@pytest.mark.parametrize("d_h,b", [(64, 32), (64, 64), (64, 128), (128, 64),
                                   (128, 128)])
def test_many_heads_per_cta(d_h, b):
    """400 heads of two tiles: every CTA passes several head changes."""
    wl = workload(d_h=d_h, block=b, N=256, B=4, H=100, race_tables=4)
    x = make_inputs(wl)
    check(wl, run(wl, x), x)


@pytest.mark.parametrize("d_h,b,nb", [(64, 64, 0), (128, 128, 0),
                                      (128, 128, 1), (64, 256, 0)])
def test_output_alignment_and_type(d_h, b, nb):
    """O at 16 bytes from a 32-byte boundary, and as fp32: the same values,
    nothing written outside."""
    wl = workload(d_h=d_h, block=b, N=b * 10, neighbor_blocks=nb)
    x = make_inputs(wl)
    a = run(wl, x)
    assert np.array_equal(a, run(wl, x, shift=16))
    f = run(wl, x, shift=16, out_fp32=1)
    assert np.array_equal(
        a, torch.from_numpy(f).to(torch.bfloat16).float().numpy())
    check(wl, a, x)
