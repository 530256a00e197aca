"""elsaa_forward_race_summaries writes to destinations of any alignment, as a
copy does: 16 bytes, 4 bytes and single bytes."""
import ctypes

import pytest
import torch

from paper_2607_20214_gb300 import build, elsaa
from paper_2607_20214_gb300.workloads import Workload, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off_a,off_b", [(0, 0), (4, 8), (2, 0), (0, 1),
                                         (3, 6)])
def test_destinations_of_any_alignment(off_a, off_b):
    build.build()
    lib = elsaa.load_library()
    wl = Workload(name="copy", B=1, H=3, N=512, d_h=64, dtype="bf16", block=64,
                  race_tables=4, recipe="plain", temperature=2.0, seed=91,
                  plane_seed=1091)
    dev = torch.device("cuda:0")
    x = {n: t.to(dev) for n, t in make_inputs(wl).items()}
    p = elsaa.params_for(wl)
    ws = elsaa.new_workspace(p, dev)
    elsaa.elsaa_forward(p, x["q"], x["k"], x["v"], x["w_sort"], x["w_race"],
                        workspace=ws)
    want = [t.contiguous().view(torch.uint8).flatten()
            for t in elsaa.elsaa_forward_race_summaries(p, ws)]
    got = [torch.zeros(w.numel() + 32, dtype=torch.uint8, device=dev)
           for w in want]
    rc = lib.elsaa_forward_race_summaries(
        ctypes.byref(p), ws.data_ptr(), ws.numel() * ws.element_size(),
        got[0].data_ptr() + off_a, got[1].data_ptr() + off_b,
        torch.cuda.current_stream(dev).cuda_stream)
    assert rc == 0
    for w, g, off in zip(want, got, (off_a, off_b)):
        assert torch.equal(g[off:off + w.numel()], w)
        assert not g[:off].any() and not g[off + w.numel():].any()
