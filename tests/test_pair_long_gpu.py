"""The CTA-pair block kernel over long ranges of blocks (about 14 per cluster,
both slots many times round), heads that begin and end inside a range, heads of
two blocks and of one: against the fp64 oracle as in test_pair_gpu.py, and the
same bits from run to run."""
import numpy as np
import pytest
import torch

from paper_2607_20214_gb300.workloads import make_inputs
from test_pair_gpu import pair_wl
from test_parity_gpu import compare, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,N,heads", [
    (17, 16384, (0, 8, 16)), (300, 512, (0, 149, 299)),
    (1000, 256, (0, 500, 999)),
])
def test_long_ranges(H, N, heads):
    wl = pair_wl(H=H, N=N, seed=81)
    x = make_inputs(wl)
    rows = np.arange(N) if N <= 512 else np.unique(np.concatenate([
        np.random.default_rng(7).choice(N, 300, replace=False),
        np.arange(N - 200, N)]))
    g = run_gpu(wl, x)
    compare(wl, g, run_oracle(wl, x, heads=[(0, h) for h in heads], rows=rows),
            label="pair H=%d N=%d" % (H, N))
    for _ in range(3):
        assert torch.equal(run_gpu(wl, x)["O_raw"], g["O_raw"])
