"""The per-example convolution statistic with few examples, whose positions are cut into parts that blocks take: one example, parts
of unequal length, every way a tile gets its rows, one layer and several in a call.

Checked against PyTorch in fp64.  Bound 1e-5 of the same statistic of absolute values: signed sums can cancel."""
import threading

import pytest
import torch

import paper_1802_06058_b200 as vgc

pytestmark = pytest.mark.gpu

SHAPES = [  # B, C, H, Cout, k, stride
    (1, 40, 56, 70, 1, 1), (1, 300, 28, 60, 1, 1), (6, 288, 24, 96, 1, 1), (3, 140, 20, 130, 1, 1),      # both tiles by TMA
    (2, 30, 28, 20, 3, 1), (1, 128, 26, 96, 3, 1), (4, 9, 30, 30, 3, 1), (3, 64, 32, 66, 3, 2), (2, 24, 44, 33, 3, 2),
    (1, 17, 40, 20, 5, 1), (2, 12, 28, 140, 7, 1), (1, 3, 64, 64, 7, 2),
    (2, 20, 33, 140, 3, 2), (1, 6, 23, 20, 5, 1), (2, 24, 25, 30, 1, 1), (1, 5, 37, 40, 4, 1),               # gathered one by one
    (30, 20, 16, 100, 3, 1),                                                                                 # enough of them
]


@pytest.mark.parametrize("layers", [1, 2])
@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("B,C,H,Cout,k,stride", SHAPES)
def test_parts(B, C, H, Cout, k, stride, accumulate, layers):
    pad = k // 2
    Ho = (H + 2 * pad - k) // stride + 1
    gen = torch.Generator("cuda").manual_seed(B * C + Cout)
    xs = [torch.randn(B, C, H, H, device="cuda", generator=gen) for _ in range(layers)]
    ds = [torch.randn(B, Cout, Ho, Ho, device="cuda", generator=gen) * 1e-3 for _ in range(layers)]
    Ss = [torch.rand(Cout, C, k, k, device="cuda", generator=gen) if accumulate else torch.full((Cout, C, k, k), -1.0, device="cuda")
          for _ in range(layers)]
    old = [S.double() if accumulate else torch.zeros_like(S, dtype=torch.float64) for S in Ss]
    size = vgc.vgc_sqgrad_conv_batch_workspace_bytes(layers, B, C, H, H, Cout, k, k, stride, stride, pad, pad, exact=True)
    ws = torch.zeros(max(256, size), dtype=torch.uint8, device="cuda")
    vgc.vgc_sqgrad_conv_exact_batch(xs, ds, (k, k), (stride, stride), (pad, pad), 0.5, Ss, accumulate, ws)
    assert int(ws[:4].view(torch.int32)) == 0
    for x, d, S, o in zip(xs, ds, Ss, old):
        cols = torch.nn.functional.unfold(x.double(), k, padding=pad, stride=stride)
        dd = d.double().reshape(B, Cout, -1)
        want = torch.einsum("bop,bip->boi", dd, cols).square().sum(0).reshape(S.shape) * 0.5 + o
        most = torch.einsum("bop,bip->boi", dd.abs(), cols.abs()).square().sum(0).reshape(S.shape) * 0.5 + o
        assert float(((S.double() - want).abs() / most).max()) < 1e-5


def test_hint_that_changes_during_calls():
    """The planning hint decides whether examples are cut up, and so which kernels can run: a call goes by one reading of it, whatever
    another thread sets meanwhile."""
    B, C, H, Cout = 2, 64, 28, 64
    gen = torch.Generator("cuda").manual_seed(3)
    x, d = torch.rand(B, C, H, H, device="cuda", generator=gen), torch.rand(B, Cout, H, H, device="cuda", generator=gen)
    cols, dd = torch.nn.functional.unfold(x.double(), 3, padding=1), d.double().reshape(B, Cout, -1)
    want = torch.einsum("bop,bip->boi", dd, cols).square().sum(0).reshape(-1)
    need = 0
    for hint in (2, 1):
        vgc.vgc_sqgrad_plan_hint(hint)
        need = max(need, vgc.vgc_sqgrad_conv_exact_workspace_bytes(B, C, H, H, Cout, 3, 3, 1, 1, 1, 1))
    ws, stop = torch.zeros(need, dtype=torch.uint8, device="cuda"), threading.Event()

    def toggle():
        hint = vgc.load_library().vgc_sqgrad_plan_hint
        while not stop.is_set():
            for _ in range(50):
                hint(2)
                hint(1)

    thread = threading.Thread(target=toggle)
    thread.start()
    try:
        worst = 0.0
        for _ in range(2000):
            S = torch.empty(Cout * C * 9, device="cuda")
            vgc.vgc_sqgrad_conv_exact(x, d, (3, 3), (1, 1), (1, 1), 1.0, S, False, ws)
            worst = max(worst, float(((S.double() - want).abs() / want).max()))
    finally:
        stop.set()
        thread.join()
        vgc.vgc_sqgrad_plan_hint(1)
    assert worst < 1e-5
