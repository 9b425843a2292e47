"""Squares and sums that leave the range of fp32, in dense layers of fewer than 32 examples on either kernel: infinite where
they are infinite, NaN where an infinite square meets a zero, and as ever in all other elements."""
import pytest
import torch

import paper_1802_06058_b200 as vgc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("B,n_in,n_out", [(1, 8192, 8192), (9, 4100, 2052), (31, 2048, 1000), (5, 64, 36), (7, 33, 65)])
def test_infinite_squares(B, n_in, n_out, accumulate):
    gen = torch.Generator("cuda").manual_seed(B)
    x, d = torch.randn(B, n_in, device="cuda", generator=gen), torch.randn(B, n_out, device="cuda", generator=gen)
    x[0, 3], x[B - 1, n_in - 2], d[B // 2, n_out - 1] = float("inf"), 1e20, -3e25       # infinite, infinite squares
    d[0, 7], x[0, 5] = 0.0, float("nan")                                                # infinity times zero; NaN stays NaN
    ws = torch.zeros(max(256, vgc.vgc_sqgrad_linear_workspace_bytes(B, n_in, n_out)), dtype=torch.uint8, device="cuda")
    old = torch.rand(n_in * n_out, device="cuda", generator=gen) if accumulate else torch.zeros(n_in * n_out, device="cuda")
    S = vgc.vgc_sqgrad_linear(x, d, 0.5, old.clone(), accumulate, ws)
    want = torch.zeros(n_out, n_in, device="cuda")
    for z in range(B):
        want += d[z].square()[:, None] * x[z].square()[None, :]
    want = old + want.reshape(-1) * 0.5
    assert int(torch.isinf(want).sum()) >= 2 * n_out - 2 and int(torch.isnan(want).sum()) >= n_out
    assert torch.equal(torch.isnan(S), torch.isnan(want)) and torch.equal(torch.isinf(S), torch.isinf(want))
    finite = torch.isfinite(want)
    assert bool(((S - want).abs()[finite] <= 2e-5 * want[finite]).all()) and int(ws[:4].view(torch.int32).item()) == 0
