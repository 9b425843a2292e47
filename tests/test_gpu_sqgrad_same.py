"""Convolutions of 3, 5 and 7 taps that keep the width (5 and 7: input rows by TMA): widths of every remainder, planes of less than a
tile's rows, channels around the edges of tiles, both statistics; sums of few terms, and of as many as make the cross terms' operands
bf16, there also at stride 2.

Checked against PyTorch in fp64.  Bound 1e-5 relative to each entry of the squared sums (all terms positive, three products per
term drop less than 2^-18 of it, an accumulator run loses less than 2e-6) and, for the per-example statistic, of the same sums
of absolute values."""
import pytest
import torch

import paper_1802_06058_b200 as vgc

pytestmark = pytest.mark.gpu

SHAPES = [  # B, C, H, W, Cout, k, pad_h
    (2, 21, 8, 8, 65, 3, 1), (2, 22, 14, 14, 130, 3, 1), (1, 64, 16, 4, 33, 3, 1), (3, 5, 7, 7, 16, 3, 1), (2, 43, 6, 10, 128, 3, 1),
    (40, 64, 14, 14, 140, 3, 1), (2, 3, 32, 32, 16, 3, 1), (2, 30, 9, 12, 20, 3, 0), (2, 30, 8, 12, 20, 3, 2),
    (2, 7, 8, 8, 65, 5, 2), (2, 8, 14, 14, 130, 5, 2), (3, 31, 17, 17, 48, 5, 2), (5, 16, 12, 12, 72, 5, 2), (1, 64, 8, 4, 129, 5, 2),
    (2, 4, 10, 10, 24, 7, 3), (2, 6, 16, 16, 130, 7, 3), (3, 3, 14, 14, 64, 7, 3), (2, 9, 9, 9, 40, 7, 3), (20, 12, 28, 28, 100, 7, 3),
    (1, 2, 16, 2, 16, 5, 2), (1, 2, 8, 6, 16, 7, 3),
]


def _inputs(B, C, H, W, Cout, k, pad_h, seed):
    Ho = H + 2 * pad_h - k + 1
    gen = torch.Generator("cuda").manual_seed(seed)
    x = torch.randn(B, C, H, W, device="cuda", generator=gen)
    d = torch.randn(B, Cout, Ho, W, device="cuda", generator=gen) * 1e-3
    return x, d


def _columns(x, k, pad_h):
    return torch.nn.functional.unfold(x.double(), k, padding=(pad_h, k // 2))


def _run(entry, need, x, d, k, pad_h, S, accumulate):
    B, C, H, W = x.shape
    size = need(B, C, H, W, d.shape[1], k, k, 1, 1, pad_h, k // 2)
    ws = torch.zeros(max(256, size), dtype=torch.uint8, device="cuda")
    entry(x, d, (k, k), (1, 1), (pad_h, k // 2), 0.5, S, accumulate, ws)
    assert int(ws[:4].view(torch.int32)) == 0
    return S


@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("B,C,H,W,Cout,k,pad_h", SHAPES)
def test_squares(B, C, H, W, Cout, k, pad_h, accumulate):
    x, d = _inputs(B, C, H, W, Cout, k, pad_h, B * C + Cout)
    S = torch.rand(Cout, C, k, k, device="cuda") if accumulate else torch.full((Cout, C, k, k), -1.0, device="cuda")
    want = torch.einsum("bop,bip->oi", d.double().reshape(B, Cout, -1).square(), _columns(x, k, pad_h).square()).reshape(S.shape) * 0.5
    if accumulate:
        want += S.double()
    _run(vgc.vgc_sqgrad_conv, vgc.vgc_sqgrad_conv_workspace_bytes, x, d, k, pad_h, S, accumulate)
    assert float(((S.double() - want).abs() / want.clamp_min(1e-30)).max()) < 1e-5


@pytest.mark.parametrize("B,C,H,W,Cout,k,pad_h", SHAPES)
def test_per_example(B, C, H, W, Cout, k, pad_h):
    x, d = _inputs(B, C, H, W, Cout, k, pad_h, B + C * Cout)
    S = torch.full((Cout, C, k, k), -1.0, device="cuda")
    cols, dd = _columns(x, k, pad_h), d.double().reshape(B, Cout, -1)
    want = torch.einsum("bop,bip->boi", dd, cols).square().sum(0).reshape(S.shape) * 0.5
    size = torch.einsum("bop,bip->boi", dd.abs(), cols.abs()).square().sum(0).reshape(S.shape) * 0.5
    _run(vgc.vgc_sqgrad_conv_exact, vgc.vgc_sqgrad_conv_exact_workspace_bytes, x, d, k, pad_h, S, False)
    assert float(((S.double() - want).abs() / size.clamp_min(1e-30)).max()) < 1e-5


@pytest.mark.parametrize("H,W,k", [(8, 8, 3), (14, 14, 3), (10, 10, 5), (9, 9, 7)])
def test_infinities_stay_where_they_are_read(H, W, k):
    """Sums that no infinite input belongs to (an example's last rows and columns, which some taps never read) are finite."""
    x, d = _inputs(2, 4, H, W, 20, k, k // 2, H)
    x[0, 1, H - 1] = float("inf")
    x[1, 2, :, W - 1] = float("inf")
    x[1, 3, 0, 0] = float("inf")
    S = torch.full((20, 4, k, k), -1.0, device="cuda")
    cols = torch.nn.functional.unfold(x.double(), k, padding=k // 2).square()
    want = torch.einsum("bop,bip->oi", d.double().reshape(2, 20, -1).square(), cols).reshape(S.shape) * 0.5
    _run(vgc.vgc_sqgrad_conv, vgc.vgc_sqgrad_conv_workspace_bytes, x, d, k, k // 2, S, False)
    finite = torch.isfinite(want)
    assert bool(finite[:, 0].all()) and not bool(finite.all()) and bool(torch.isfinite(S[finite]).all())
    assert float(((S.double() - want)[finite].abs() / want[finite]).max()) < 1e-5


@pytest.mark.parametrize("C,H,W,Cout,k,stride", [(64, 4, 8, 512, 3, 1), (64, 8, 16, 512, 3, 2), (3, 8, 16, 512, 7, 2), (32, 4, 8, 512, 5, 1),
                                                 (16, 4, 8, 512, 7, 1), (64, 2, 16, 512, 3, 1), (64, 16, 2, 512, 3, 1)])
def test_few_terms(C, H, W, Cout, k, stride):
    """Sums of 32 terms, most of them one term's: all parts are tf32 there.  One slice, twelve instructions that truncate (2^-23 of the sum
    each at most), two cross terms of 2^-11 of the product with 11 bits read of a part (2^-21 each), 2^-22 dropped, two roundings
    (2^-24 each); bf16 copies add up to 2^-18."""
    gen = torch.Generator("cuda").manual_seed(C + k)
    x = torch.randn(1, C, H, W, device="cuda", generator=gen)
    d = torch.randn(1, Cout, H // stride, W // stride, device="cuda", generator=gen)
    d *= torch.exp(2 * torch.randn(d.shape, device="cuda", generator=gen))
    ws = torch.zeros(max(256, vgc.vgc_sqgrad_conv_workspace_bytes(1, C, H, W, Cout, k, k, stride, stride, k // 2, k // 2)), dtype=torch.uint8, device="cuda")
    S = torch.zeros(Cout, C * k * k, device="cuda")
    vgc.vgc_sqgrad_conv(x, d, (k, k), (stride, stride), (k // 2, k // 2), 1.0, S, False, ws)
    cols = torch.nn.functional.unfold(x.double(), k, padding=k // 2, stride=stride)[0]
    want = d.double().reshape(Cout, -1).square() @ cols.square().t()
    some = want > 0                                                          # (taps that only ever read padding)
    assert torch.equal(S > 0, some)
    assert float(((S.double() - want).abs() / want)[some].max()) < 12 * 2.0 ** -23 + 2 * 2.0 ** -21 + 2.0 ** -22 + 2 * 2.0 ** -24


@pytest.mark.parametrize("C,H,Cout,k,stride,B", [(320, 8, 1024, 3, 1, 15), (320, 8, 1024, 3, 1, 16), (320, 6, 1000, 3, 1, 28), (320, 6, 1000, 3, 1, 29),
                                                 (320, 16, 1024, 3, 2, 15), (320, 16, 1024, 3, 2, 16), (320, 12, 1024, 3, 2, 29), (64, 16, 1024, 7, 2, 15),
                                                 (64, 16, 1024, 7, 2, 16), (64, 8, 1000, 5, 1, 15), (65, 8, 1000, 5, 1, 16), (64, 10, 1024, 5, 1, 10),
                                                 (64, 10, 1024, 5, 1, 11), (48, 8, 1024, 7, 1, 15), (49, 8, 1024, 7, 1, 16), (48, 6, 900, 7, 1, 29)])
def test_many_terms(C, H, Cout, k, stride, B):
    """About 1024 terms in long accumulator runs, from where on the cross terms take bf16 copies, in every form of wide tiles."""
    x = torch.randn(B, C, H, H, device="cuda", generator=torch.Generator("cuda").manual_seed(B + C))
    d = torch.randn(B, Cout, H // stride, H // stride, device="cuda", generator=torch.Generator("cuda").manual_seed(k)) * 1e-3
    ws = torch.zeros(vgc.vgc_sqgrad_conv_workspace_bytes(B, C, H, H, Cout, k, k, stride, stride, k // 2, k // 2), dtype=torch.uint8, device="cuda")
    S = torch.full((Cout, C * k * k), -1.0, device="cuda")
    vgc.vgc_sqgrad_conv(x, d, (k, k), (stride, stride), (k // 2, k // 2), 0.5, S, False, ws)
    cols = torch.nn.functional.unfold(x.double(), k, padding=k // 2, stride=stride).square()
    want = torch.einsum("bop,bip->oi", d.double().reshape(B, Cout, -1).square(), cols) * 0.5
    assert int(ws[:4].view(torch.int32)) == 0 and float(((S.double() - want).abs() / want).max()) < 1e-5
