"""A workspace that starts on any 4-byte boundary: the bits of one that starts on a 256-byte boundary, whichever way partial tiles
are added up.  (Layers that are repacked into the workspace need 16 bytes: TMA reads them there.)"""
import pytest
import torch

import paper_1802_06058_b200 as vgc

pytestmark = pytest.mark.gpu

CONV = [  # B, C, H, Cout, k, stride, per-example
    (32, 128, 28, 128, 3, 1, False), (9, 544, 16, 48, 3, 2, False), (4, 64, 16, 40, 1, 1, False), (16, 16, 16, 48, 5, 1, False),
    (1, 24, 64, 30, 4, 1, False), (2, 64, 28, 64, 3, 1, True), (6, 288, 24, 96, 1, 1, True), (33, 12, 16, 130, 3, 1, True),
]


def _workspaces(need):
    need = max(256, need)
    yield torch.zeros(need, dtype=torch.uint8, device="cuda")
    for at in (4, 8, 12, 20):
        ws = torch.zeros(need + 32, dtype=torch.uint8, device="cuda")[at:at + need]
        assert ws.data_ptr() % 16 == at % 16
        yield ws


@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("B,C,H,Cout,k,stride,exact", CONV)
def test_conv(B, C, H, Cout, k, stride, exact, accumulate):
    pad = k // 2
    Ho = (H + 2 * pad - k) // stride + 1
    gen = torch.Generator("cuda").manual_seed(B + C)
    x, d = torch.randn(B, C, H, H, device="cuda", generator=gen), torch.randn(B, Cout, Ho, Ho, device="cuda", generator=gen)
    query = vgc.vgc_sqgrad_conv_exact_workspace_bytes if exact else vgc.vgc_sqgrad_conv_workspace_bytes
    call = vgc.vgc_sqgrad_conv_exact if exact else vgc.vgc_sqgrad_conv
    want = None
    for ws in _workspaces(query(B, C, H, H, Cout, k, k, stride, stride, pad, pad)):
        S = torch.ones(Cout * C * k * k, device="cuda")
        call(x, d, (k, k), (stride, stride), (pad, pad), 0.5, S, accumulate, ws)
        want = S if want is None else want
        assert torch.equal(S, want) and int(ws[:4].view(torch.int32)) == 0


@pytest.mark.parametrize("B,n_in,n_out", [(1024, 512, 512), (3000, 260, 132), (700, 901, 903)])
def test_dense(B, n_in, n_out):
    gen = torch.Generator("cuda").manual_seed(B)
    x, d = torch.randn(B, n_in, device="cuda", generator=gen), torch.randn(B, n_out, device="cuda", generator=gen)
    want = None
    for ws in _workspaces(vgc.vgc_sqgrad_linear_workspace_bytes(B, n_in, n_out)):
        S = vgc.vgc_sqgrad_linear(x, d, 0.5, torch.ones(n_in * n_out, device="cuda"), True, ws)
        want = S if want is None else want
        assert torch.equal(S, want) and int(ws[:4].view(torch.int32)) == 0
