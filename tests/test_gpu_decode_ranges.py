"""The decoder at the sizes where its forms and ranges change: buffers around one block's least range (2048 elements),
tiles that span two tensors, tensors too small or too many for the exact form, indices crowded at one end (the interpolating
search has to fall back), and word counts on either side of the lines between flat, scatter and dense.  Values are powers of
two within seven binades and the scale is one, so that every sum is exact in fp32: bit for bit, whatever the order."""
import numpy as np
import pytest
import torch

import oracle
import paper_1802_06058_b200 as vgc
from gpu_harness import Guarded, random_offsets
from paper_1802_06058_b200 import workloads

pytestmark = pytest.mark.gpu
F32 = np.float32


def _check(n, offs, msgs):
    triples = [(w if w.numel() else torch.zeros(4, dtype=torch.int32, device="cuda"),
                torch.tensor([w.numel()], dtype=torch.int32, device="cuda"), e) for w, e in msgs]
    host = [(w.cpu().numpy().view(np.uint32), e.cpu().numpy()) for w, e in msgs]
    for overwrite in (False, True):
        gu = Guarded(n, fill=float("nan") if overwrite else 0.5)
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        vgc.vgc_decode_accumulate(triples, vgc.offsets_tensor(offs), 1.0, gu.t, st, overwrite=overwrite)
        gu.check("u")
        ref = np.zeros(n, F32) if overwrite else np.full(n, 0.5, F32)
        oracle.decode_accumulate(host, offs, 1.0, ref)
        assert int(st.item()) == 0
        assert np.array_equal(gu.t.cpu().numpy().view(np.uint32), ref.view(np.uint32))


def _message(n, offs, density, seed, lo=0.0, hi=1.0):
    mask = torch.zeros(n, dtype=torch.bool, device="cuda")
    a, b = int(n * lo), max(int(n * lo) + 1, int(n * hi))
    gen = torch.Generator("cuda").manual_seed(seed)
    mask[a:b] = torch.empty(b - a, device="cuda").uniform_(generator=gen) < density
    words, exps = workloads.random_message(n, offs, density, seed + 1, "cuda", index_mask=mask)
    return words, torch.full_like(exps, -1) - (exps & 1)


@pytest.mark.parametrize("n", [1, 7, 2047, 2048, 2049, 4099, 2048 * 444 + 3])
@pytest.mark.parametrize("density", [0.004, 0.3])
@pytest.mark.parametrize("W", [1, 3, 9])
def test_small_ranges(n, density, W):
    offs = random_offsets(np.random.default_rng(n), n, min(n, 6))
    _check(n, offs, [_message(n, offs, density, 10 * w + n) for w in range(W)])


@pytest.mark.parametrize("sizes", [[100_000, 5, 900_000], [33_333, 3, 2, 1, 400_001, 17, 90_001], [64] * 3000, [0, 70_001, 0, 0, 1_500_002],
                                   [0] * 600 + [40_000, 2] + [0] * 900 + [1, 30_000, 0, 5, 0]])
def test_tensor_borders_anywhere(sizes):
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint32)
    n = int(offs[-1])
    _check(n, offs, [_message(n, offs, 0.1, 50 + w) for w in range(8)])


@pytest.mark.parametrize("W", [2, 20, 64])
@pytest.mark.parametrize("density", [0.9, 0.02])
def test_crowded_indices(W, density):
    n = 3_000_001
    offs = random_offsets(np.random.default_rng(W), n, 5)
    msgs = [_message(n, offs, density, 70 + w, *((0.0, 0.02) if w % 2 else (0.97, 0.985))) for w in range(W)]
    _check(n, offs, msgs)


@pytest.mark.parametrize("n", [1_000_003, 5_000_003])
@pytest.mark.parametrize("words_per_element", [1 / 17.5, 1 / 15, 1 / 8.6, 1 / 7.4])
def test_either_side_of_the_lines(n, words_per_element):
    offs = random_offsets(np.random.default_rng(4), n, 4)
    _check(n, offs, [_message(n, offs, words_per_element / 3, 90 + w) for w in range(3)])


@pytest.mark.parametrize("lengths", [[20_000] + [0] * 7, [30_000, 15_001, 15_000, 14_999, 1, 33], [5, 9_000, 0, 70_000, 2, 35_000] * 10, [31], [33, 16]])
def test_flat_messages_of_unequal_lengths(lengths):
    """Few words, added: the pieces of every message are taken once, whatever the lengths beside it."""
    n, offs = 8_000_003, np.array([0, 5, 70_000, 8_000_003], np.uint32)
    msgs = []
    for w, c in enumerate(lengths):
        words, exps = _message(n, offs, 1.3 * c / n + 1e-6, 300 + w)
        msgs.append((words[:c].clone(), exps))
    assert [m[0].numel() for m in msgs] == lengths
    _check(n, offs, msgs)


def test_flat_form_costs_what_the_words_cost():
    """Seven short messages beside a long one must not cost what seven long ones would (every piece of a message that ran
    out of words once took a warp's turn: 5 to 13 times the long message's own time)."""
    n = 30_000_000
    offs = np.array([0, n], np.uint32)

    def time(lengths):
        msgs = [_message(n, offs, c / n, 400 + w) for w, c in enumerate(lengths)]
        triples = [(m, torch.tensor([m.numel()], dtype=torch.int32, device="cuda"), e) for m, e in msgs]
        u, st, o = torch.zeros(n, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda"), vgc.offsets_tensor(offs)
        best = float("inf")
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                vgc.vgc_decode_accumulate(triples, o, 1.0, u, st)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    alone = time([1_500_000])
    assert time([1_500_000] + [200] * 63) < 3.0 * alone


@pytest.mark.parametrize("sizes", [[50_000] + [64, 64] * 40 + [300_000], [1] * 2000 + [70_000], [0] * 50 + [40_000] + [0] * 55 + [3, 0, 0, 5] * 200 + [9_001],
                                   list(range(1, 900)) + [200_003], [500] * 1200 + [7]])
@pytest.mark.parametrize("W", [3, 8, 40, 64])
def test_form_is_chosen_tensor_by_tensor(sizes, W):
    """More tensors in a block's range and in a tile than any fixed number, with a scale that is no power of two.  A tensor
    whose exponents lie close together is scale * the exact sum, its neighbour whose exponents do not is the sequential sum:
    both bit for bit."""
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint32)
    n, K, scale = int(offs[-1]), len(sizes), np.float32(1.0 / 7)
    apart = np.random.default_rng(K).random(K) < 0.3                       # tensors that take the ordered form
    host, dev = [], []
    for w in range(W):
        words, exps = _message(n, offs, 1.2 / W, 500 + w)
        exps = np.where(apart, -5 - 25 * (w % 2), exps.cpu().numpy()).astype(np.int32)
        host.append((words.cpu().numpy().view(np.uint32), exps))
        dev.append((words, torch.tensor([words.numel()], dtype=torch.int32, device="cuda"), torch.from_numpy(exps).cuda()))
    ordered = np.repeat(apart, sizes)
    for overwrite in (False, True):
        u0 = np.zeros(n, F32) if overwrite else np.random.default_rng(1).standard_normal(n).astype(F32)
        gu = Guarded(n)
        gu.t.copy_(torch.from_numpy(u0))
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        vgc.vgc_decode_accumulate(dev, vgc.offsets_tensor(offs), float(scale), gu.t, st, overwrite=overwrite)
        gu.check("u")
        sequential, exact = u0.copy(), np.zeros(n, F32)
        oracle.decode_accumulate(host, offs, float(scale), sequential)
        oracle.decode_accumulate([(m, np.where(apart, 0, e).astype(np.int32)) for m, e in host], offs, 1.0, exact)
        touched = np.zeros(n, bool)
        for m, _ in host:
            touched[m >> 4] = True
        scaled = np.where(touched & (exact != 0), u0 + exact * scale, u0)   # (float32: each operation rounded once)
        want = np.where(ordered, sequential, scaled).astype(F32)
        assert int(st.item()) == 0
        got = gu.t.cpu().numpy()
        assert np.array_equal(got, want), (np.flatnonzero(got != want)[:5], got[got != want][:5], want[got != want][:5])
