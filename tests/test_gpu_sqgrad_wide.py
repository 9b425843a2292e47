"""Tiles of 192 columns (and their neighbours of 128) of the convolution statistic: edges of tiles, short and long reductions.

The contraction is checked against PyTorch in fp64.  Bound 1e-5 relative to each entry: all terms are positive, three products
per term drop less than 2^-18 of it, and an accumulator run of at most 96 truncating instructions loses less than 2e-6."""
import pytest
import torch

import paper_1802_06058_b200 as vgc

pytestmark = pytest.mark.gpu

SHAPES = [  # B, C, H, Cout, k
    (2, 129, 8, 65, 1), (2, 192, 8, 100, 1), (2, 65, 8, 192, 1), (1, 193, 6, 130, 1),      # one tile and its edges
    (3, 512, 14, 128, 1), (3, 128, 14, 512, 1), (2, 400, 12, 260, 1), (4, 1030, 7, 72, 1),  # several, ragged last one
    (40, 300, 28, 140, 1),                                                                  # long reduction, shared tiles
    (2, 43, 8, 72, 3), (2, 64, 28, 140, 3), (1, 21, 8, 65, 3), (2, 22, 14, 130, 3),          # gathered: 387, 576, 189 and 198 columns
    (3, 4, 16, 64, 7),                                                                      # 196 columns, gathered one by one
]


@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("B,C,H,Cout,k", SHAPES)
def test_wide_tiles(B, C, H, Cout, k, accumulate):
    gen = torch.Generator("cuda").manual_seed(B * C + Cout)
    x = torch.randn(B, C, H, H, device="cuda", generator=gen)
    d = torch.randn(B, Cout, H, H, device="cuda", generator=gen) * 1e-3
    S = torch.rand(Cout, C, k, k, device="cuda", generator=gen) if accumulate else torch.full((Cout, C, k, k), -1.0, device="cuda")
    cols = torch.nn.functional.unfold(x.double(), k, padding=k // 2).square()
    want = torch.einsum("bop,bip->oi", d.double().reshape(B, Cout, -1).square(), cols).reshape(S.shape) * 0.5
    if accumulate:
        want += S.double()
    ws = torch.zeros(max(256, vgc.vgc_sqgrad_conv_workspace_bytes(B, C, H, H, Cout, k, k, 1, 1, k // 2, k // 2)),
                     dtype=torch.uint8, device="cuda")
    vgc.vgc_sqgrad_conv(x, d, (k, k), (1, 1), (k // 2, k // 2), 0.5, S, accumulate, ws)
    assert int(ws[:4].view(torch.int32)) == 0
    assert float(((S.double() - want).abs() / want).max()) < 1e-5
