"""How the per-example statistic cuts few long examples into parts, seen through the workspace it asks for: the best of all part
lengths, found without trying each of them."""
import time

import paper_1802_06058_b200 as vgc

SMS, SLICE, ROWS, COMBINE, PARTS_COMBINE = 148, 32, 128, 4, 14


def _up(a, b):
    return -(-a // b)


def _partial_tiles(M, N, examples, slices, tile_n, layers):
    """Bytes of partial tiles of one launch alone on the GPU, by trying every part length."""
    tiles = _up(N, tile_n) * _up(M, ROWS) * layers
    units, k_slices = tiles * examples, examples * slices
    waves = _up(tiles, SMS)
    blocks = _up(tiles, waves)
    even_blocks = min(units, SMS)
    even = _up(units, even_blocks) * slices + COMBINE < _up(tiles, blocks) * k_slices
    if even:
        blocks = even_blocks
    slot = ROWS * (192 if tile_n > 128 else 128) * 4
    if slices > 1:
        best = (_up(units, blocks) if even else _up(tiles, blocks) * examples) * slices + (PARTS_COMBINE if even else 0)
        parts = 0
        for q in range(1, slices):
            n = units * _up(slices, q)
            if n <= 2 * SMS and _up(n, SMS) * (q + 5) + PARTS_COMBINE < best:
                best, parts = _up(n, SMS) * (q + 5) + PARTS_COMBINE, n
        if parts:
            return parts * slot
    total, upt = (units, examples) if even else (tiles, 1)
    q, r = divmod(total, blocks)
    shared = any((b * q + min(b, r)) % upt for b in range(1, blocks))
    return 2 * blocks * slot if shared else 0


def _workspace(layers, B, C, H, Cout, k):
    """3x3, 5x5 and 7x7 at stride 1 with the padding that keeps the size, planes of whole vectors (nothing is repacked)."""
    N, slices = C * k * k, _up(H * H, SLICE)
    narrow = (N, Cout) if Cout <= 64 and N > Cout else (Cout, N)
    need = [256 + _partial_tiles(*narrow, B, slices, 128, layers), 256 + _partial_tiles(Cout, N, B, slices, 192, layers)]
    if k > 3:
        need.append(256 + _partial_tiles(Cout, N, B, slices, 192 // k * k, layers))
    return _up(max(need) + 256, 256) * 256


def test_parts_of_examples():
    seen = set()
    for layers in (1, 3, 8):
        for B in (1, 2, 3, 6, 9, 17, 40, 150):
            for C, Cout in ((3, 16), (17, 65), (64, 64), (128, 130), (300, 48), (40, 300)):
                for H in (8, 12, 28, 40, 64, 112, 224):
                    for k in (3, 5, 7):
                        got = vgc.vgc_sqgrad_conv_batch_workspace_bytes(layers, B, C, H, H, Cout, k, k, 1, 1, k // 2, k // 2, exact=True)
                        assert got == _workspace(layers, B, C, H, Cout, k), (layers, B, C, H, Cout, k)
                        seen.add(got)
    assert len(seen) > 50


def test_long_examples_are_planned_as_fast_as_short_ones():
    """8.4 million slices an example: trying every part length took 0.1 s a query."""
    vgc.load_library()
    start = time.perf_counter()
    for _ in range(50):
        assert vgc.vgc_sqgrad_conv_exact_workspace_bytes(1, 1, 16384, 16384, 16, 3, 3, 1, 1, 1, 1) > 256
    assert time.perf_counter() - start < 1.0
