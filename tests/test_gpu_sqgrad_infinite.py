"""Squares and sums at and beyond the end of fp32's range.  Beyond it, in dense layers of fewer than 32 examples on either kernel: infinite
where they are infinite, NaN where an infinite square meets a zero, and as ever in all other elements.  Before it: finite in every form."""
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


@pytest.mark.parametrize("B,C,H,Cout,k,stride", [(32, 64, 16, 128, 3, 1), (32, 64, 14, 128, 3, 1), (8, 64, 32, 66, 3, 2), (8, 3, 64, 64, 7, 2),
                                                 (16, 32, 16, 64, 5, 1), (16, 32, 16, 64, 7, 1), (8, 128, 16, 128, 1, 1), (8, 128, 7, 128, 1, 1),
                                                 (32, 33, 17, 64, 4, 1), (128, 1024, 0, 1024, 0, 0), (512, 1024, 0, 1024, 0, 0), (1024, 512, 0, 512, 0, 0)])
def test_largest_finite_squares(B, C, H, Cout, k, stride):
    """A square that is finite in fp32 and tf32 and would round to infinity in bf16 (3.398e38), on either side: its sums are finite,
    like all others within 1e-5."""
    gen = torch.Generator("cuda").manual_seed(B + C)
    dense, pad = k == 0, k // 2
    Ho = 0 if dense else (H + 2 * pad - k) // stride + 1
    x = torch.randn((B, C) if dense else (B, C, H, H), device="cuda", generator=gen)
    d = torch.randn((B, Cout) if dense else (B, Cout, Ho, Ho), device="cuda", generator=gen)
    for large, small in ((x, d), (d, x)):
        a, b = large.clone(), small * 1e-6
        a.view(B, -1)[B // 2, 5] = 1.8433e19
        xx, dd = (a, b) if large is x else (b, a)
        S = torch.zeros(Cout * C * max(1, k * k), device="cuda")
        if dense:
            ws = torch.zeros(max(256, vgc.vgc_sqgrad_linear_workspace_bytes(B, C, Cout)), dtype=torch.uint8, device="cuda")
            vgc.vgc_sqgrad_linear(xx, dd, 1.0, S, False, ws)
            want = dd.double().square().t() @ xx.double().square()
        else:
            ws = torch.zeros(max(256, vgc.vgc_sqgrad_conv_workspace_bytes(B, C, H, H, Cout, k, k, stride, stride, pad, pad)), dtype=torch.uint8, device="cuda")
            vgc.vgc_sqgrad_conv(xx, dd, (k, k), (stride, stride), (pad, pad), 1.0, S, False, ws)
            cols = torch.nn.functional.unfold(xx.double(), k, padding=pad, stride=stride).square()
            want = torch.einsum("bop,bip->oi", dd.double().reshape(B, Cout, -1).square(), cols)
        assert int(ws[:4].view(torch.int32)) == 0 and bool(torch.isfinite(want.float()).all())
        assert float(((S.double() - want.reshape(-1)).abs() / want.reshape(-1)).max()) < 1e-5
