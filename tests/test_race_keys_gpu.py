"""RACE key summaries A, B of the tensor-core kernels against 64 bits, at
table counts that fill a row half unevenly and lengths that leave tiles and
chunks partly empty. Features are rounded to bf16 (2^-9) after factors from
an approximate tanh (2^-11 each): |A - A_ref| <= 2^-7 A_ref and
|B - B_ref| <= 2^-7 sum phi |v|."""
import pytest
import torch

from paper_2607_20214_gb300 import build, elsaa
from paper_2607_20214_gb300.workloads import Workload, make_inputs

pytestmark = pytest.mark.gpu


def phi64(k, w):
    u = torch.tanh(torch.einsum("bhnd,hlgd->bhnlg", k.double(), w.double()))
    s = torch.sigmoid(2 * u)
    out = torch.ones(s.shape[:-1] + (1,), dtype=s.dtype, device=s.device)
    for b in range(s.shape[-1]):
        out = torch.cat([out * (1 - s[..., b:b + 1]), out * s[..., b:b + 1]],
                        -1)
    return out.flatten(3)


@pytest.mark.parametrize("d_h", [64, 128])
@pytest.mark.parametrize("L,N,B,H", [
    (1, 32, 1, 1), (3, 96, 1, 2), (4, 160, 1, 3), (5, 4128, 1, 1),
    (7, 288, 2, 2), (8, 1920, 1, 3), (8, 128, 2, 80), (9, 64, 1, 1),
    (13, 544, 1, 2), (16, 2080, 1, 2), (16, 8192, 1, 1), (16, 384, 3, 60),
])
def test_summaries(d_h, L, N, B, H):
    build.build()
    wl = Workload("keys", B=B, H=H, N=N, d_h=d_h, dtype="bf16", block=32,
                  race_tables=L, seed=71, plane_seed=1071)
    x = make_inputs(wl, device="cuda")
    p = elsaa.params_for(wl)
    ws = elsaa.new_workspace(p, x["q"].device)
    ws.fill_(0xFF)  # NaN wherever a partial is left out
    elsaa.elsaa_forward(p, x["q"], x["k"], x["v"], x["w_sort"], x["w_race"],
                        workspace=ws)
    A, Bm = elsaa.elsaa_forward_race_summaries(p, ws)
    elsaa.elsaa_check_status(ws)
    f = phi64(x["k"], x["w_race"])
    ref_a = f.sum(2)
    assert ((A - ref_a).abs() <= 2 ** -7 * ref_a).all()
    ref_b = f.transpose(2, 3) @ x["v"].double()
    scale = f.transpose(2, 3) @ x["v"].double().abs()
    assert ((Bm - ref_b).abs() <= 2 ** -7 * scale).all()
