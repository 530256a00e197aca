"""Where the scan of a short call has a launch of its own: beyond 1024 counts
(tiles of 128 rows times bins) per order, unless the call has at most 152 CTAs
and 2048 counts. Orders are exact on both sides of the line."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2607_20214_gb300 import build, elsaa
from paper_2607_20214_gb300.workloads import Workload, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,N,bits,apart", [
    (4, 8192, 5, True), (32, 1024, 8, True), (8, 4096, 6, True),
    (8, 4096, 5, False), (32, 512, 8, False), (1, 8192, 5, False),
    (9, 1024, 8, False), (10, 1024, 8, True), (1, 8224, 5, True),
    (2, 4096, 6, False), (3, 4096, 6, True),
])
def test_scan_launch_and_orders(heads, N, bits, apart):
    build.build()
    wl = Workload(name="scan", B=1, H=heads, N=N, d_h=64, dtype="bf16",
                  block=32, race_tables=4, temperature=2.0, sort_bits=bits,
                  seed=95, plane_seed=1095)
    x = make_inputs(wl)
    xd = {n: t.cuda() for n, t in x.items()}
    p = elsaa.params_for(wl)
    ws = elsaa.new_workspace(p, torch.device("cuda:0"))
    pq = torch.full((1, heads, N), -1, dtype=torch.int32, device="cuda")
    pk = torch.full_like(pq, -1)
    elsaa.elsaa_profile_start()
    elsaa.elsaa_forward(p, xd["q"], xd["k"], xd["v"], xd["w_sort"],
                        xd["w_race"], workspace=ws, perm_q=pq, perm_k=pk)
    torch.cuda.synchronize()
    prof = elsaa.elsaa_profile_stop()
    elsaa.elsaa_check_status(ws)
    assert ("sort_scan" in prof) == apart, prof
    for h in sorted({0, heads - 1}):
        for name, got in (("q", pq), ("k", pk)):
            keys, _ = orc.sort_keys(orc.to_numpy32(x[name][0, h]),
                                    orc.to_numpy32(x["w_sort"][h]),
                                    wl.gray_order)
            assert np.array_equal(got[0, h].cpu().numpy(),
                                  orc.stable_argsort(keys)), (h, name)
