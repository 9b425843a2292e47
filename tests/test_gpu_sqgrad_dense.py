"""Dense layers on either side of the lines between the kernels (multiply-adds, examples, sizes TMA cannot address) and at
the edges of their tiles: one example, one slice, the last slice of one and of two accumulators, one tile and several per
block, ragged borders; written and added.  Reference: fp64 matmul of the squares.  Bound: 1e-5 relative (the library's own);
written and added results agree to one fp32 addition exactly."""
import pytest
import torch

import paper_1802_06058_b200 as vgc
from gpu_harness import Guarded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n_in,n_out", [
    (1, 8192, 8192), (9, 4100, 2052), (31, 2048, 1000), (33, 1028, 1092), (64, 4096, 4096), (64, 5000, 3004),   # one slice to many tiles
    (255, 516, 516), (256, 512, 1000), (257, 512, 516), (512, 260, 516), (511, 2048, 132), (513, 512, 516),     # one and two accumulators
    (128, 1000, 1024), (70, 2364, 512), (300, 68, 1028), (130, 9472, 128), (130, 9476, 128),                   # 64 columns: at most 74 tiles of 128
    (1, 3, 5), (5, 32, 33), (64, 63, 129), (65, 64, 64), (129, 1000, 10), (200, 333, 257), (1024, 40, 36), (1025, 33, 65),
    (128, 1031, 1009)])
def test_dense(B, n_in, n_out):
    gen = torch.Generator("cuda").manual_seed(B + n_in)
    x = torch.randn(B, n_in, device="cuda", generator=gen).clamp_(min=0)
    d = torch.randn(B, n_out, device="cuda", generator=gen) * 1e-3
    x[:, 0] = 0
    nb = max(256, vgc.vgc_sqgrad_linear_workspace_bytes(B, n_in, n_out))
    scale = 1.0 / (B * B)
    want = (d.double().square().t() @ x.double().square()).mul_(scale).reshape(-1)
    S, T, ws = Guarded(n_in * n_out, fill=float("nan")), Guarded(n_in * n_out), Guarded(nb, torch.uint8, fill=0)
    T.t.normal_(generator=gen).abs_().mul_(float(want.mean()))
    old = T.t.clone()
    for _ in range(2):                                           # again, right behind the first call
        vgc.vgc_sqgrad_linear(x, d, scale, S.t, ws=ws.t)
    vgc.vgc_sqgrad_linear(x, d, scale, T.t, accumulate=True, ws=ws.t)
    assert int(ws.t[:4].view(torch.int32).item()) == 0
    for g in (S, T, ws):
        g.check()
    assert bool(((S.t.double() - want).abs() <= 1e-5 * want).all())
    if B > 1024:      # this kernel adds old and new in fp64 and rounds once: at most the rounding of S apart, 2^-24 of it, and
        both = old.double() + S.t.double()                       # the rounding of either sum, 2^-24 each: 3 * 2^-24 in all
        assert bool(((T.t.double() - both).abs() <= 3 * 2.0 ** -24 * both).all())
    else:
        assert torch.equal(T.t, old + S.t)


@pytest.mark.parametrize("B,n_in,n_out", [
    (127, 1031, 1009), (640, 901, 901), (768, 333, 257), (769, 333, 257), (769, 500, 256), (768, 500, 256), (1024, 20, 300),
    (900, 1301, 1301), (1024, 701, 701),                                                        # CUDA cores: one launch or a split reduction
    (576, 512, 512), (1024, 512, 512), (2048, 64, 64), (5000, 260, 36)])                        # many partial tiles per tile
def test_long_reductions(B, n_in, n_out):
    test_dense(B, n_in, n_out)


@pytest.mark.parametrize("B,n_in,n_out", [(1100, 333, 257), (1300, 33, 35), (640, 901, 901), (3000, 512, 512)])
def test_added_is_one_fp32_addition(B, n_in, n_out):
    """Long reductions, too: what is added is the written result, rounded once (a compressor step with s in v counts on it)."""
    x, d = torch.randn(B, n_in, device="cuda"), torch.randn(B, n_out, device="cuda")
    ws = torch.zeros(vgc.vgc_sqgrad_linear_workspace_bytes(B, n_in, n_out), dtype=torch.uint8, device="cuda")
    S, T = torch.empty(n_in * n_out, device="cuda"), torch.rand(n_in * n_out, device="cuda")
    vgc.vgc_sqgrad_linear(x, d, 1.0 / B, S, ws=ws)
    want = T + S
    vgc.vgc_sqgrad_linear(x, d, 1.0 / B, T, accumulate=True, ws=ws)
    assert torch.equal(T, want)


@pytest.mark.parametrize("B", [191, 192, 193, 224, 255, 256, 257, 512])
@pytest.mark.parametrize("n_in,n_out", [(1024, 1024), (1000, 132), (4096, 1300), (132, 2052)])
def test_cross_terms_in_bf16(B, n_in, n_out):
    """Around the number of examples from which the two cross terms take bf16 copies (each a 2^-11 of the product, the copies good
    to 2^-9 of it): narrow and full tiles, edges of tiles and slices.  Bound 1e-5 of every entry, all of whose terms are positive."""
    gen = torch.Generator("cuda").manual_seed(B + n_in)
    x = torch.randn(B, n_in, device="cuda", generator=gen)
    d = torch.randn(B, n_out, device="cuda", generator=gen) * 1e-3
    ws = torch.zeros(max(256, vgc.vgc_sqgrad_linear_workspace_bytes(B, n_in, n_out)), dtype=torch.uint8, device="cuda")
    want = (d.double().square().t() @ x.double().square()) * 0.5
    for accumulate in (False, True):
        S = torch.rand(n_out, n_in, device="cuda", generator=gen) * 1e-4 if accumulate else torch.full((n_out, n_in), -1.0, device="cuda")
        full = want + S.double() if accumulate else want
        vgc.vgc_sqgrad_linear(x, d, 0.5, S, accumulate, ws)
        assert int(ws[:4].view(torch.int32)) == 0
        assert float(((S.double() - full).abs() / full).max()) < 1e-5
