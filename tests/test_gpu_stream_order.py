"""Arrays of the caller's that the kernel just ahead on the stream writes, with nothing between it and the call that reads
them.  That kernel is one of the library's, which lets the next one start under its own end: whatever the next one reads too
early is seen here as the array's old content.  Both contents are valid arguments, so a stale read gives a wrong answer only."""
import numpy as np
import pytest
import torch

import paper_1802_06058_b200 as vgc
from gpu_harness import noise_gs, random_offsets
from paper_1802_06058_b200 import workloads

pytestmark = pytest.mark.gpu


class Written:
    """An int32 array that a kernel of the library (vgc_unpack_indices, which copies any ascending words) writes in turn."""

    def __init__(self, *contents):
        n = contents[0].size
        self.t = torch.zeros(n, dtype=torch.int32, device="cuda")
        self.n, self.status = torch.tensor([n], dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        self.packed = []
        for c in contents:
            words = torch.from_numpy(c.astype(np.uint32).view(np.int32)).cuda()
            p, b = torch.zeros(vgc.vgc_pack_bound_bytes(n), dtype=torch.uint8, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
            ws = torch.zeros(vgc.vgc_pack_workspace_bytes(n), dtype=torch.uint8, device="cuda")
            vgc.vgc_pack_indices(words, self.n, p, b, self.status, ws)
            self.packed.append(p)

    def write(self, which):
        vgc.vgc_unpack_indices(self.packed[which], self.n, self.t, self.status)


@pytest.mark.parametrize("n,K", [(40_000, 9), (2_000_003, 700), (2_000_003, 3000)])
def test_offsets_written_just_ahead(n, K):
    rng = np.random.default_rng(K)
    offs = [random_offsets(rng, n, K) for _ in range(2)]
    written = Written(*offs)
    g, s = noise_gs(n, 4, seed=K)
    ws = torch.empty(vgc.vgc_compress_workspace_bytes(n, K), dtype=torch.uint8, device="cuda")
    # dense, scatter (written) and flat (added) decodes
    sets = [[(m, torch.tensor([m.numel()], dtype=torch.int32, device="cuda"), e)
             for m, e in (workloads.random_message(n, offs[0], d, w, "cuda") for w in range(3))] for d in (0.2, 0.01)]

    def step(which, out, r, v, u):
        r.zero_(), v.zero_()
        for t in u:
            t.fill_(0.5)
        ahead(which)
        vgc.vgc_compress(g, s, r, v, written.t, 2.0, 0.999, out, ws)
        for i, (msgs, overwrite) in enumerate([(sets[0], True), (sets[0], False), (sets[1], True), (sets[1], False)]):
            ahead(which)
            vgc.vgc_decode_accumulate(msgs, written.t, 1.0, u[i], written.status, overwrite=overwrite)

    def buffers():
        return vgc.MessageBuffers(n, K, n), torch.empty(n, device="cuda"), torch.empty(n, device="cuda"), [torch.empty(n, device="cuda") for _ in range(4)]

    def ahead(which):
        written.write(which)
        torch.cuda.synchronize()

    want = []
    for which in (0, 1):
        b = buffers()
        step(which, *b)
        want.append((b[0].read(), b[1], b[2], b[3]))

    def ahead(which):                                                # noqa: F811 -- the other content first, then no pause
        written.write(1 - which)
        torch.cuda.synchronize()
        written.write(which)

    for turn in range(6):
        b = buffers()
        step(turn & 1, *b)
        got, ref = b[0].read(), want[turn & 1]
        assert np.array_equal(got["group_exp"], ref[0]["group_exp"]) and np.array_equal(got["words"], ref[0]["words"])
        assert torch.equal(b[1], ref[1]) and torch.equal(b[2], ref[2])
        # (where two words meet in an element, the order of their additions is free in the sparse forms)
        assert all(torch.allclose(x, y, rtol=2.0 ** -22, atol=1e-8) for x, y in zip(b[3], ref[3]))
    assert int(written.status.item()) == 0


def _alternate(call, inputs, results):
    """call(input, result) for the inputs one after another without a pause, against the same with the stream idle before each."""
    want = []
    for i in inputs:
        torch.cuda.synchronize()
        call(i, results[0])
        torch.cuda.synchronize()
        want.append(results[0].clone())
    for _ in range(4):
        for i, r in zip(inputs, results):
            call(i, r)
        for w, r in zip(want, results):
            assert torch.equal(w, r)


# padded planes (7 x 7, pitch 196 bytes) with stride 1 and 2, subsampled planes, planes merged channel by channel, gathered rows
@pytest.mark.parametrize("C,H,Cout,k,stride,pad,exact", [(64, 7, 96, 3, 1, 1, False), (64, 7, 96, 3, 1, 1, True), (32, 14, 64, 3, 2, 1, False),
                                                         (128, 28, 96, 1, 2, 0, False), (256, 7, 96, 1, 1, 0, False),
                                                         (48, 9, 40, 5, 1, 2, False), (64, 28, 64, 3, 1, 1, False)])
def test_layers_change_between_calls_on_one_workspace(C, H, Cout, k, stride, pad, exact):
    B, Ho = 16, (H + 2 * pad - k) // stride + 1
    geo = (B, C, H, H, Cout, k, k, stride, stride, pad, pad)
    need = (vgc.vgc_sqgrad_conv_exact_workspace_bytes if exact else vgc.vgc_sqgrad_conv_workspace_bytes)(*geo)
    ws = torch.zeros(need, dtype=torch.uint8, device="cuda")
    inputs = [(torch.randn(B, C, H, H, device="cuda"), torch.randn(B, Cout, Ho, Ho, device="cuda")) for _ in range(4)]
    fn = vgc.vgc_sqgrad_conv_exact if exact else vgc.vgc_sqgrad_conv
    _alternate(lambda i, S: fn(*i, (k, k), (stride, stride), (pad, pad), 1.0, S, ws=ws), inputs,
               [torch.empty(Cout * C * k * k, device="cuda") for _ in inputs])
    assert int(ws[:4].view(torch.int32).item()) == 0


@pytest.mark.parametrize("B,n_in,n_out", [(32, 64, 40), (16, 1024, 4096), (600, 96, 64)])
def test_layer_input_written_just_ahead(B, n_in, n_out):
    """x of a layer is the result of the call ahead (CUDA cores, tensor cores, long reductions)."""
    ws = torch.zeros(max(vgc.vgc_sqgrad_linear_workspace_bytes(8, n_in, B), vgc.vgc_sqgrad_linear_workspace_bytes(B, n_in, n_out)),
                     dtype=torch.uint8, device="cuda")
    x, d = torch.empty(B * n_in, device="cuda"), torch.randn(B, n_out, device="cuda")
    inputs = [(torch.randn(8, n_in, device="cuda"), torch.randn(8, B, device="cuda")) for _ in range(4)]

    def call(i, S):
        vgc.vgc_sqgrad_linear(*i, 1.0, x, ws=ws)
        vgc.vgc_sqgrad_linear(x.view(B, n_in), d, 1.0, S, ws=ws)

    _alternate(call, inputs, [torch.empty(n_in * n_out, device="cuda") for _ in inputs])


def test_stream_packed_just_ahead():
    n = 300_000
    status, ws = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros(vgc.vgc_pack_workspace_bytes(n), dtype=torch.uint8, device="cuda")
    packed, nbytes = torch.zeros(vgc.vgc_pack_bound_bytes(n), dtype=torch.uint8, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    inputs = []
    for seed in range(4):
        words, _ = workloads.random_message(4 * n, np.array([0, 4 * n], np.uint32), 0.2, seed, "cuda")
        inputs.append((words[:n].clone(), torch.tensor([min(n, words.numel())], dtype=torch.int32, device="cuda")))

    def call(i, back):
        back.zero_()
        vgc.vgc_pack_indices(*i, packed, nbytes, status, ws)
        vgc.vgc_unpack_indices(packed, i[1], back, status)

    back = [torch.zeros(n, dtype=torch.int32, device="cuda") for _ in inputs]
    _alternate(call, inputs, back)
    assert all(torch.equal(b[:i[0].numel()], i[0]) for b, i in zip(back, inputs)) and int(status.item()) == 0
