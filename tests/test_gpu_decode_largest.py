"""The decoder on the largest buffer, 2^28 elements: there every 28-bit index is an element, the filler of a partly filled
piece of words included.  Few words (the flat and scatter forms), message lengths that are no multiples of a piece, none at
all, and more messages than one launch takes.  u is the oracle's where words point and untouched everywhere else."""
import numpy as np
import pytest
import torch

import oracle
import paper_1802_06058_b200 as vgc

pytestmark = pytest.mark.gpu
N = vgc.VGC_MAX_PARAMS


def _messages(lengths, hybrid):
    msgs = []
    for w, c in enumerate(lengths):
        rng = np.random.default_rng(c + w)
        idx = np.unique(np.append(rng.integers(1, N - 1, c), [0, N - 1])).astype(np.uint32)
        idx = idx[idx.size - c:] if w % 3 == 1 else idx[:c]              # the last element among them, or not
        low = rng.integers(0, 16, idx.size).astype(np.uint32)
        words = idx << 4 | (low & 8 if hybrid else low)
        msgs.append((words, np.array([-3 + w % 2, vgc.VGC_EXP_NONE if c == 0 else -4, -5], np.int32)))
    return msgs


@pytest.mark.parametrize("hybrid", [False, True])
@pytest.mark.parametrize("lengths", [[333], [1, 500, 0, 77], [40 + 3 * w for w in range(70)]])
def test_largest_buffer(hybrid, lengths):
    offs = np.array([0, 1000, N - 4096, N], np.uint32)
    msgs = _messages(lengths, hybrid)
    dev = [(torch.from_numpy(np.append(m, np.uint32(0)).view(np.int32)).cuda(), torch.tensor([m.size], dtype=torch.int32, device="cuda"),
            torch.from_numpy(e).cuda()) for m, e in msgs]
    want = np.zeros(N, np.float32)                                # (pages nobody touches cost nothing)
    if hybrid:
        oracle.decode_hybrid([m for m, _ in msgs], 0.25, 0.5, want)
    else:
        oracle.decode_accumulate(msgs, offs, 0.5, want)
    touched = np.unique(np.concatenate([m >> 4 for m, _ in msgs])).astype(np.int64)
    at = torch.from_numpy(touched).cuda()
    u = torch.empty(N, device="cuda")
    for overwrite in (False, True):
        u.fill_(7.0 if overwrite else 0.0)
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        if hybrid:
            vgc.vgc_decode_accumulate_hybrid([m[:2] for m in dev], 0.25, 0.5, u, st, overwrite=overwrite)
        else:
            vgc.vgc_decode_accumulate(dev, vgc.offsets_tensor(offs), 0.5, u, st, overwrite=overwrite)
        assert int(st.item()) == 0
        # sums of a few powers of two within eleven binades: exact in fp32, whatever the order
        assert np.array_equal(u[at].cpu().numpy(), want[touched])
        u[at] = 0.0
        assert int(torch.count_nonzero(u)) == 0
