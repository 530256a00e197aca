"""The top-k selection on the tensor cores (bf16, key blocks of a multiple
of 128): exactly the oracle's key sets at every candidate count, at the ends
of the range of k, with ties, and for rows that only the canonical chain can
decide (zero, tiny and huge rows)."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2607_20214_gb300 import build, elsaa
from paper_2607_20214_gb300.workloads import Workload, make_inputs

pytestmark = pytest.mark.gpu


def check(wl, x):
    build.build()
    dev = torch.device("cuda:0")
    p = elsaa.params_for(wl)
    xd = {n: t.to(dev) for n, t in x.items()}
    ws = elsaa.new_workspace(p, dev)
    elsaa.elsaa_forward(p, xd["q"], xd["k"], xd["v"], xd["w_sort"],
                        xd["w_race"], workspace=ws)
    keys = elsaa.elsaa_forward_selected_keys(p, ws)
    elsaa.elsaa_check_status(ws)
    got = keys.cpu().numpy()
    for (b, h), r in orc.forward(x, orc.params_from_workload(wl)).items():
        bad = np.nonzero((got[b, h][r["rows"]] != r["sel"]).any(axis=1))[0]
        assert bad.size == 0, (wl, b, h, r["rows"][bad[:8]])


def workload(**kw):
    base = dict(name="topk_tc", B=1, H=2, N=1024, d_h=64, dtype="bf16",
                block=128, race_tables=4, recipe="plain", temperature=2.0,
                seed=51, plane_seed=1051, selector=1, topk=64, topk_blocks=2)
    base.update(kw)
    return Workload(**base)


@pytest.mark.parametrize("d_h,b,c,k", [
    (64, 128, 1, 1), (64, 128, 1, 127), (128, 128, 1, 128),
    (128, 128, 2, 1), (64, 128, 2, 255), (128, 128, 2, 256),
    (128, 128, 3, 7), (64, 128, 3, 383), (128, 128, 4, 511),
    (64, 256, 1, 33), (64, 256, 2, 256), (64, 384, 1, 200),
    (64, 512, 1, 300),
])
def test_sets_at_the_edges(d_h, b, c, k):
    wl = workload(d_h=d_h, block=b, topk_blocks=c, topk=k, N=b * max(c, 3))
    check(wl, make_inputs(wl))


@pytest.mark.parametrize("c,k", [(1, 50), (2, 100), (4, 300)])
def test_ties(c, k):
    """Small integers: every row has many equal scores at its threshold."""
    wl = workload(topk_blocks=c, topk=k, sort_bits=2)
    x = make_inputs(wl)
    for n in ("q", "k"):
        x[n] = torch.round(x[n].float().clamp(-1.5, 1.5)).to(torch.bfloat16)
    check(wl, x)


def test_duplicate_keys():
    wl = workload(topk=100)
    x = make_inputs(wl)
    x["k"][:, :, 1::2] = x["k"][:, :, ::2]
    check(wl, x)


@pytest.mark.parametrize("scale", [0.0, 1e-20, 1e-38, 3e18])
def test_rows_for_the_chain_alone(scale):
    """Rows whose squared norm underflows, overflows or is zero."""
    wl = workload(H=1, topk=90)
    x = make_inputs(wl)
    x["q"][:, :, ::3] *= scale
    check(wl, x)
    x = make_inputs(wl)
    x["k"][:, :, ::5] *= min(scale, 3e18)
    check(wl, x)


def test_uneven_scores():
    """Score distributions far from a normal one: heavy tails, two far
    groups, one dominant element."""
    wl = workload(d_h=128, H=3, topk=77)
    x = make_inputs(wl)
    k = x["k"].float()
    k[:, 0] *= torch.exp(2.0 * torch.randn(k[:, 0].shape[:2]))[..., None]
    k[:, 1, ::4] += 6.0
    k[:, 2, :, 0] *= 300.0
    x["k"] = k.to(torch.bfloat16)
    check(wl, x)
