"""The streaming kernel of both compressors at the sizes where its partition changes: one parameter, around one block's
least share (2048), around one tile per block (4096 x 296 blocks), several rounds of the second kernel,
tensors that begin and end in the middle of tiles and blocks; and a
captured launch replayed, which finds what it left in the workspace.  Bit-exact against the oracle (whole numbers; fp32 operations rounded
one by one on both sides)."""
import numpy as np
import pytest
import torch

import oracle
import paper_1802_06058_b200 as vgc
from gpu_harness import GpuCompressor, OracleCompressor, assert_same_message, assert_same_state, noise_gs, random_offsets

pytestmark = pytest.mark.gpu

FULL = 296 * 4096


@pytest.mark.parametrize("n,K,alpha", [(1, 1, 2.0), (2047, 3, 2.0), (2049, 1, 2.0), (FULL - 3, 11, 2.0), (FULL + 130, 2, 1.0),
                                       (2 * FULL + 1, 1500, 2.0), (4_500_001, 5, 0.0), (4_500_004, 400, 0.0)])
def test_compress_over_block_borders(n, K, alpha):
    offs = random_offsets(np.random.default_rng(n), n, K)
    gpu, cpu = GpuCompressor(n, offs), OracleCompressor(n, offs)
    for t in range(2):
        g, s = noise_gs(n, 4, seed=700 + t)
        got = gpu.step(g, s, alpha, 0.999)
        assert_same_message(got, cpu.step(g.cpu().numpy(), s.cpu().numpy(), alpha, 0.999))
        assert_same_state(gpu, cpu)


@pytest.mark.parametrize("n,tau", [(1, 1e-3), (2049, 1e-3), (1 << 18, 0.0), (FULL + 5, 1e-3), (4_500_001, 0.0)])
def test_hybrid_over_block_borders(n, tau):
    r, v = torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda")
    rc, vc = np.zeros(n, np.float32), np.zeros(n, np.float32)
    out = vgc.HybridMessageBuffers(n, n, with_mask=True)
    ws = torch.empty(vgc.vgc_compress_hybrid_workspace_bytes(n), dtype=torch.uint8, device="cuda").fill_(0x5A)
    for t in range(2):
        g, s = noise_gs(n, 4, seed=800 + t)
        vgc.vgc_compress_hybrid(g, s, r, v, 0.5, 0.999, tau, out, ws)
        got = out.read()
        want = oracle.compress_hybrid(g.cpu().numpy(), s.cpu().numpy(), rc, vc, 0.5, 0.999, tau)
        assert got["dev_status"] == 0 and got["nnz"] == want.nnz
        assert np.array_equal(got["words"], want.words) and np.array_equal(got["mask"], want.mask)
        assert np.array_equal(r.cpu().numpy().view(np.uint32), rc.view(np.uint32))
        assert np.array_equal(v.cpu().numpy().view(np.uint32), vc.view(np.uint32))


def test_replayed_launch():
    n, K = 700_001, 9
    offs = random_offsets(np.random.default_rng(3), n, K)
    gpu, cpu = GpuCompressor(n, offs), OracleCompressor(n, offs)
    g, s = noise_gs(n, 4, seed=900)
    gpu.step(g, s, 2.0, 0.999)
    cpu.step(g.cpu().numpy(), s.cpu().numpy(), 2.0, 0.999)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        vgc.vgc_compress(g, s, gpu.r, gpu.v, gpu.offs_dev, 2.0, 0.999, gpu.out, gpu.ws)
    for t in range(4):
        g2, s2 = noise_gs(n, 4, seed=901 + t)
        g.copy_(g2)
        s.copy_(s2)
        graph.replay()
        assert_same_message(gpu.out.read(), cpu.step(g2.cpu().numpy(), s2.cpu().numpy(), 2.0, 0.999))
        assert_same_state(gpu, cpu)
