"""Kernels that only short calls take, at the edges of their rules: the scan
fused into the scatter (at most 32768 rows and 2048 tile-bin counts per
order; orders are exact), the copy of the RACE summaries to destinations
that are only 4-byte aligned (bytes are exact), and the CUDA-core block
kernel with 8 queries per CTA (grids of fewer than 152 tiles of 32; fp32
tolerance 1e-4, as for every fp32 output against the oracle)."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2607_20214_gb300 import build, elsaa
from paper_2607_20214_gb300.workloads import Workload, make_inputs

pytestmark = pytest.mark.gpu


def workload(**kw):
    base = dict(name="short", B=1, H=1, N=256, d_h=64, dtype="bf16", block=32,
                race_tables=4, temperature=2.0, seed=91, plane_seed=1091)
    base.update(kw)
    return Workload(**base)


def run(wl, x, **out):
    build.build()
    p = elsaa.params_for(wl)
    xd = {n: t.cuda() for n, t in x.items()}
    ws = elsaa.new_workspace(p, torch.device("cuda:0"))
    o = elsaa.elsaa_forward(p, xd["q"], xd["k"], xd["v"], xd["w_sort"],
                            xd["w_race"], workspace=ws, **out)
    elsaa.elsaa_check_status(ws)
    return p, ws, o.float().cpu().numpy()


# tiles of 128 rows, 2^bits bins: 1 tile, a ragged last tile, 2048 counts
# and the next size up, 32768 rows and the next size up
@pytest.mark.parametrize("heads,N,bits", [
    (1, 32, 5), (3, 160, 5), (2, 1024, 8), (2, 1152, 8), (1, 8192, 5),
    (1, 8224, 5), (2, 224, 0), (5, 992, 1), (32, 1024, 5), (33, 1024, 5),
])
def test_orders(heads, N, bits):
    wl = workload(H=heads, N=N, sort_bits=bits)
    x = make_inputs(wl)
    pq = torch.full((1, heads, N), -1, dtype=torch.int32, device="cuda")
    pk = torch.full_like(pq, -1)
    run(wl, x, perm_q=pq, perm_k=pk)
    for h in sorted({0, heads // 2, heads - 1}):
        for name, got in (("q", pq), ("k", pk)):
            keys, _ = orc.sort_keys(orc.to_numpy32(x[name][0, h]),
                                    orc.to_numpy32(x["w_sort"][h]),
                                    wl.gray_order)
            assert np.array_equal(got[0, h].cpu().numpy(),
                                  orc.stable_argsort(keys)), (h, name)


@pytest.mark.parametrize("L,bits", [(1, 1), (3, 4), (16, 4)])
@pytest.mark.parametrize("sa,sb", [(0, 0), (1, 0), (0, 1), (2, 3)])
def test_summaries_unaligned(L, bits, sa, sb):
    wl = workload(H=2, race_tables=L, race_bits=bits)
    p, ws, _ = run(wl, make_inputs(wl))
    A, Bm = elsaa.elsaa_forward_race_summaries(p, ws)
    ba = torch.full((A.numel() + 8,), float("nan"), device="cuda")
    bb = torch.full((Bm.numel() + 8,), float("nan"), device="cuda")
    va, vb = ba[sa:sa + A.numel()], bb[sb:sb + Bm.numel()]
    elsaa.elsaa_forward_race_summaries(p, ws, race_A=va.view(A.shape),
                                       race_B=vb.view(Bm.shape))
    assert torch.equal(va.view(A.shape), A)
    assert torch.equal(vb.view(Bm.shape), Bm)
    assert torch.isnan(ba[:sa]).all() and torch.isnan(ba[sa + A.numel():]).all()
    assert torch.isnan(bb[:sb]).all() and torch.isnan(bb[sb + Bm.numel():]).all()


# 8 queries per CTA up to 151 tiles of 32, 32 from 152 on
@pytest.mark.parametrize("kw", [
    dict(N=32), dict(N=96, d_h=32), dict(N=160, d_h=128, H=3),
    dict(N=1024, race_tables=16), dict(N=256, block=128, race_bits=6),
    dict(N=256, block=64, race_bits=1, race_tables=3),
    dict(N=192, block=64, race_bits=5, race_tables=5),
    dict(N=512, block=64, neighbor_blocks=1),
    dict(N=512, block=64, selector=1, topk=48, topk_blocks=3),
    dict(N=4832), dict(N=4864), dict(N=4896),
])
def test_block_kernel_small_grids(kw):
    wl = workload(dtype="fp32", **kw)
    x = make_inputs(wl)
    _, _, o = run(wl, x)
    for (b, h), r in orc.forward(x, orc.params_from_workload(wl)).items():
        assert np.abs(o[b, h] - r["O"]).max() <= 1e-4, (b, h)
