"""vgc_step_host: staging buffers of their own (copies run beside the kernels), shared between the layers and with g (copies
and kernels take turns), a message whose counters do not lie side by side, and calls from several threads on streams of
their own; staging in memory that the kernels of earlier layers write.  All give what the device calls give, bit for bit."""
import ctypes
import threading

import numpy as np
import pytest
import torch

import paper_1802_06058_b200 as vgc
from paper_1802_06058_b200 import workloads

pytestmark = pytest.mark.gpu
B, SIZES = 64, [(1024, 512), (512, 256), (256, 12)]


class Step:
    def __init__(self, seed, staging, B=B):
        specs = [workloads.LayerSpec(f"fc{i}", "fc", a, b) for i, (a, b) in enumerate(SIZES)]
        offs = workloads.group_offsets(specs)
        self.n, self.K = int(offs[-1]), len(specs)
        self.offs = vgc.offsets_tensor(offs)
        ins = [workloads.layer_inputs(sp, B, 1, 0, seed, i, "relu_normal", 1e-3, "cuda") for i, sp in enumerate(specs)]
        g = torch.cat([workloads.mean_gradient(sp, x, d) for sp, (x, d) in zip(specs, ins)])
        self.ws = torch.zeros(max(vgc.vgc_sqgrad_linear_workspace_bytes(B, sp.cin, sp.cout) for sp in specs) + 256,
                              dtype=torch.uint8, device="cuda")
        self.wc = torch.empty(vgc.vgc_compress_workspace_bytes(self.n, self.K), dtype=torch.uint8, device="cuda")
        self.s, self.r, self.v = (torch.zeros(self.n, device="cuda") for _ in range(3))
        for (x, d), lo, hi in zip(ins, offs[:-1].tolist(), offs[1:].tolist()):
            vgc.vgc_sqgrad_linear(x, d, 1.0 / B ** 2, self.s[lo:hi], ws=self.ws)
        out = vgc.MessageBuffers(self.n, self.K, self.n)
        vgc.vgc_compress(g, self.s, self.r, self.v, self.offs, 2.0, 0.999, out, self.wc)
        self.want = out.read()
        self.B = B
        self.g_dev = torch.empty(self.n, device="cuda")
        in_ws = self.ws[1 << 20:self.ws.numel() // 4 * 4].view(torch.float32)     # past the status word and what small layers need
        if staging == "g in the workspace":
            self.g_dev = in_ws[:self.n]
        room = self.g_dev if staging == "with g" else torch.empty(2 * B * 1024, device="cuda")
        self.layers = []
        for x, d in ins:
            if staging == "last layer in the workspace" and d.shape[1] == SIZES[-1][1]:
                xd, dd = in_ws[:x.numel()].view_as(x), in_ws[x.numel():x.numel() + d.numel()].view_as(d)
            elif staging not in ("shared", "with g"):
                xd, dd = torch.empty_like(x), torch.empty_like(d)
            else:
                xd, dd = room[:x.numel()].view_as(x), room[x.numel():x.numel() + d.numel()].view_as(d)
            self.layers.append({"is_conv": 0, "B": B, "C": x.shape[1], "Cout": d.shape[1], "x_host": x.cpu().pin_memory(),
                                "delta_host": d.cpu().pin_memory(), "x_dev": xd, "delta_dev": dd})
        self.g_host = g.cpu().pin_memory()
        self.words, self.counters = torch.zeros(self.n, dtype=torch.int32), torch.zeros(4, dtype=torch.int32)

    def check(self, out, stream=None):
        s, r, v = torch.full_like(self.s, float("nan")), torch.zeros_like(self.r), torch.zeros_like(self.v)
        torch.cuda.synchronize()
        got = vgc.vgc_step_host(self.layers, self.g_host, self.g_dev, s, r, v, self.offs, 2.0, 0.999, 1.0 / self.B ** 2, out, self.words,
                                self.counters, self.ws, self.wc, stream=stream)
        w = self.want
        assert got == (w["nnz"], w["n_criterion"], w["n_dropped"], 0)
        assert np.array_equal(self.words[:got[0]].numpy().view(np.uint32), w["words"])
        assert torch.equal(s, self.s) and torch.equal(r, self.r) and torch.equal(v, self.v)


@pytest.mark.parametrize("staging", ["own", "shared", "with g"])
def test_staging(staging):
    step = Step(3, staging)
    out = vgc.MessageBuffers(step.n, step.K, step.n)
    for _ in range(3):
        out.counters.zero_()
        step.check(out)


@pytest.mark.parametrize("staging", ["g in the workspace", "last layer in the workspace"])
def test_staging_over_memory_that_earlier_kernels_write(staging):
    """The first layers (1100 examples) leave partial tiles all over the workspace; what is copied there for a later use
    must not arrive before they are done."""
    step = Step(5, staging, B=1100)
    assert step.ws.numel() > (1 << 20) + 4 * step.n
    out = vgc.MessageBuffers(step.n, step.K, step.n)
    for _ in range(5):
        out.counters.zero_()
        step.check(out)


def test_counters_apart():
    step = Step(4, "own")

    class Apart(vgc.MessageBuffers):
        def struct(self):
            m, c = super().struct(), self.far.data_ptr()
            m.nnz, m.n_criterion, m.n_dropped, m.dev_status = c, c + 64, c + 128, c + 192
            return m

    out = Apart(step.n, step.K, step.n)
    out.far = torch.zeros(64, dtype=torch.int32, device="cuda")
    assert isinstance(out.struct(), ctypes.Structure)
    step.check(out)


def test_threads():
    steps = [Step(10 + i, "own") for i in range(3)]
    torch.cuda.synchronize()
    failed = []

    def work(step):
        try:
            stream = torch.cuda.Stream()
            out = vgc.MessageBuffers(step.n, step.K, step.n)
            for _ in range(5):
                out.counters.zero_()
                step.check(out, stream)
        except BaseException as e:  # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=work, args=(s,)) for s in steps]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[0]


@pytest.mark.parametrize("sizes,pinned,shift", [([(1024, 512), (256, 12)], "both", 0), ([(1024, 512), (256, 12)], "both", 1),
                                                ([(1024, 512), (256, 12)], "words", 0), ([(2048, 1024), (64, 12)], "both", 0)])
def test_message_goes_home_by_a_kernel_or_by_copies(sizes, pinned, shift):
    """Page-locked results (written by a kernel up to 2^18 words), at an odd place, the counters in ordinary memory, a longer message."""
    specs = [workloads.LayerSpec(f"fc{i}", "fc", a, b) for i, (a, b) in enumerate(sizes)]
    offs = workloads.group_offsets(specs)
    n, K = int(offs[-1]), len(specs)
    ins = [workloads.layer_inputs(sp, B, 1, 0, 5, i, "relu_normal", 1e-3, "cuda") for i, sp in enumerate(specs)]
    g = torch.cat([workloads.mean_gradient(sp, x, d) for sp, (x, d) in zip(specs, ins)])
    ws = torch.zeros(max(vgc.vgc_sqgrad_linear_workspace_bytes(B, sp.cin, sp.cout) for sp in specs) + 256, dtype=torch.uint8, device="cuda")
    wc = torch.empty(vgc.vgc_compress_workspace_bytes(n, K), dtype=torch.uint8, device="cuda")
    s, r, v = (torch.zeros(n, device="cuda") for _ in range(3))
    for (x, d), lo, hi in zip(ins, offs[:-1].tolist(), offs[1:].tolist()):
        vgc.vgc_sqgrad_linear(x, d, 1.0 / B ** 2, s[lo:hi], ws=ws)
    out = vgc.MessageBuffers(n, K, n)
    vgc.vgc_compress(g, s, r, v, vgc.offsets_tensor(offs), 2.0, 0.999, out, wc)
    want = out.read()
    assert (want["nnz"] > 1 << 18) == (sizes[0][0] == 2048)
    layers = [{"is_conv": 0, "B": B, "C": x.shape[1], "Cout": d.shape[1], "x_host": x.cpu().pin_memory(), "delta_host": d.cpu().pin_memory(),
               "x_dev": torch.empty_like(x), "delta_dev": torch.empty_like(d)} for x, d in ins]
    words = torch.full((n + 8,), -1, dtype=torch.int32).pin_memory()[shift:]
    counters = torch.zeros(4, dtype=torch.int32)
    if pinned == "both":
        counters = counters.pin_memory()
    out2 = vgc.MessageBuffers(n, K, n)
    got = vgc.vgc_step_host(layers, g.cpu().pin_memory(), torch.empty_like(g), torch.empty_like(s), torch.zeros_like(r), torch.zeros_like(v),
                            vgc.offsets_tensor(offs), 2.0, 0.999, 1.0 / B ** 2, out2, words, counters, ws, wc)
    assert got == (want["nnz"], want["n_criterion"], want["n_dropped"], 0)
    assert np.array_equal(words[:want["nnz"]].numpy().view(np.uint32), want["words"])
    assert bool((words[want["nnz"]:] == -1).all())


@pytest.mark.parametrize("place", ["whole", "begins page-locked", "counters off by two bytes", "words off by two bytes"])
def test_results_where_a_kernel_cannot_write(place):
    """Results that are page-locked only in part, or lie on no word boundary, are copied: the number of launches tells which way they
    went."""
    step, launches = Step(7, "own"), vgc.vgc_kernel_launch_count

    def launched(words, counters):
        step.words, step.counters = words, counters
        before = launches()
        step.check(vgc.MessageBuffers(step.n, step.K, step.n))
        return launches() - before

    by_copies = launched(step.words, step.counters)                          # ordinary memory
    room = torch.zeros(4 * step.n + 3 * 4096, dtype=torch.uint8)
    first = -room.data_ptr() % 4096
    base, more = memoryview(room.numpy())[first:], torch.zeros(64, dtype=torch.uint8).pin_memory()
    locked = (4 * step.want["nnz"] // 4096 + 1) * 4096                       # the message fits, the buffer does not
    assert locked + 4096 < 4 * step.n and step.want["nnz"] < 1 << 18
    if not place.startswith("begins"):
        locked = 4 * step.n + 4096
    at = [2 if place.startswith(what) else 0 for what in ("words", "counters")]
    rt = torch.cuda.cudart()
    assert rt.cudaHostRegister(room.data_ptr() + first, locked, 0) == rt.cudaError.success
    try:
        count = launched(torch.frombuffer(base[at[0]:at[0] + 4 * step.n], dtype=torch.int32),
                         torch.frombuffer(memoryview(more.numpy())[at[1]:at[1] + 16], dtype=torch.int32))
    finally:
        torch.cuda.synchronize()
        assert rt.cudaHostUnregister(room.data_ptr() + first) == rt.cudaError.success
    assert count - by_copies == (1 if place == "whole" else 0)
