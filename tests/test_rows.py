"""The quotient that tells a position's row in an output plane: plain C++, compiled and run here over widths up to 2^30 and, for
each, the first and last position of rows up to the last one that 31-bit positions reach."""
import os
import subprocess

import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "vgc_rows.cuh"
static bool row_ok(uint64_t width, const vgc::RowDivisor &d, uint64_t row)
{
    const uint64_t first = row * width, last = first + width - 1 < (1ull << 31) ? first + width - 1 : (1ull << 31) - 1;
    if (vgc::row_of((uint32_t)first, d.magic, d.shift) == row && vgc::row_of((uint32_t)last, d.magic, d.shift) == row) return true;
    printf("width %llu row %llu\n", (unsigned long long)width, (unsigned long long)row);
    return false;
}
static bool width_ok(uint64_t width, bool all)
{
    const vgc::RowDivisor d = vgc::row_divisor((uint32_t)width);
    const uint64_t rows = ((1ull << 31) - 1) / width + 1;              // of 31-bit positions
    for (uint64_t row = 0; row < rows; row += all || row < 70 || row + 70 > rows ? 1 : 1 + rows / 997)
        if (!row_ok(width, d, row)) return false;
    return row_ok(width, d, rows - 1);
}
int main()
{
    for (uint64_t width = 2; width < 40000; ++width)
        if (!width_ok(width, width == 2048 || width == 4096 || width == 4100)) return 1;
    for (int l = 2; l <= 30; ++l)
        for (int off = -3; off <= 3; ++off)
            if ((1ll << l) + off >= 2 && !width_ok((1ll << l) + off, false)) return 1;
    for (uint64_t width = 40001; width < (1u << 30); width += 77777)
        if (!width_ok(width, false)) return 1;
    return 0;
}
"""


def test_rows_of_positions(tmp_path):
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(PROGRAM)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-I",
                    os.path.join(ROOT, "paper_1802_06058_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    done = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert done.returncode == 0, done.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("side,k,stride,exact", [(4096, 3, 1, False), (4096, 5, 1, False), (4096, 7, 1, False), (2048, 4, 1, False),
                                                 (4096, 7, 2, False), (4096, 4, 1, True)])
def test_large_planes(side, k, stride, exact):
    """Planes whose positions times width pass 2^32, by every way a tile gets its rows.  Bound 1e-5 of sums of positive terms."""
    import paper_1802_06058_b200 as vgc
    pad = (k - 1) // 2
    out = (side + 2 * pad - k) // stride + 1
    gen = torch.Generator("cuda").manual_seed(side + k)
    x = torch.rand(1, 1, side, side, device="cuda", generator=gen)
    d = torch.rand(1, 2, out, out, device="cuda", generator=gen)
    S = torch.zeros(2, 1, k, k, device="cuda")
    need = (vgc.vgc_sqgrad_conv_exact_workspace_bytes if exact else vgc.vgc_sqgrad_conv_workspace_bytes)(1, 1, side, side, 2, k, k, stride, stride, pad, pad)
    ws = torch.zeros(max(256, need), dtype=torch.uint8, device="cuda")
    (vgc.vgc_sqgrad_conv_exact if exact else vgc.vgc_sqgrad_conv)(x, d, (k, k), (stride, stride), (pad, pad), 1.0, S, False, ws)
    assert int(ws[:4].view(torch.int32)) == 0
    xp = torch.nn.functional.pad(x[0, 0].double(), (pad, pad + k, pad, pad + k))
    for kh in range(k):
        for kw in range(k):
            xs = xp[kh:kh + (out - 1) * stride + 1:stride, kw:kw + (out - 1) * stride + 1:stride]
            for o in range(2):
                want = float((d[0, o].double() * xs).sum() ** 2 if exact else (d[0, o].double() * xs).square().sum())
                assert abs(float(S[o, 0, kh, kw]) - want) < 1e-5 * want
