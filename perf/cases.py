"""The work that users of this library give it, as cases that can be timed.

A case is one pass through the public entry points, as a training program calls them once per step (or per layer):

  step      one worker step on the device: squared-gradient sums of every dense layer, compress, decode of W messages
  host      the same up to the message, from pinned host buffers (vgc_step_host)
  conv      the squared-gradient sums of one convolution (both statistics)
  net       the squared-gradient sums of a whole convolutional network, layers of one shape in one call
  compress  one compressor step over a flat buffer
  hybrid    one compressor step of the hybrid algorithm and the decode of W such messages
  decode    decode of W messages into the dense update (added or written)
  coder     index compression of a message for the wire and its inverse

``listed`` holds the sizes of the benchmark configurations and ragged ones between them; ``draw`` gives others from the
same ranges.  Compressor states are those of the middle of a training run: residuals and variances have been
accumulating for different numbers of steps, so that every pass sends about the same share of the parameters.
"""
import math

import numpy as np
import torch

import paper_1802_06058_b200 as vgc
from paper_1802_06058_b200 import workloads as wl

ALPHA, ZETA = 2.0, 0.999
DEV = "cuda"


def listed():
    return [
        # one small dense layer, 4 workers: launches and host work are all there is
        {"name": "dense_step", "kind": "step", "widths": "256-128", "B": 32, "W": 4, "density": 0.01, "fused": False},
        # a small MLP with a narrow last layer, 8 workers: what a first experiment looks like
        {"name": "mlp_step", "kind": "step", "widths": "784-1024-1024-10", "B": 128, "W": 8, "density": 0.01, "fused": False},
        # the same network driven from host memory, message back on the host
        {"name": "mlp_host", "kind": "host", "widths": "784-1024-1024-10", "B": 128, "density": 0.01},
        # one 3x3 layer, called on its own as a backward hook does
        {"name": "conv_3x3", "kind": "conv", "C": 128, "H": 28, "Cout": 128, "k": 3, "stride": 1, "pad": 1, "B": 32,
         "exact": False, "accumulate": False},
        # the per-example statistic, accumulated straight into v
        {"name": "conv_exact", "kind": "conv", "C": 256, "H": 14, "Cout": 256, "k": 3, "stride": 1, "pad": 1, "B": 32,
         "exact": True, "accumulate": True},
        # every layer of an ImageNet-sized network: the largest piece of a step
        {"name": "resnet50_sqgrad", "kind": "net", "h": 224, "B": 32},
        # that network's parameters, message of about one word per hundred parameters
        {"name": "resnet50_compress", "kind": "compress", "net": "resnet50", "n": 25502912, "K": 54, "density": 0.01,
         "mask": False},
        # the largest buffers: the dense layers of VGG-16, squared sums added straight into v, long messages
        {"name": "vgg16_dense_step", "kind": "step", "widths": "25088-4096-4096-1000", "B": 64, "W": 4, "density": 0.03,
         "fused": True},
        # hybrid algorithm on a ragged medium-sized buffer
        {"name": "hybrid_step", "kind": "hybrid", "n": 3274635, "K": 1, "W": 8, "density": 0.005},
        # dense update of 8 workers whose messages are long
        {"name": "decode_dense", "kind": "decode", "net": "resnet50", "n": 25502912, "K": 54, "W": 8, "density": 0.05,
         "overwrite": True},
        # many workers with short messages, added to what is there
        {"name": "decode_sparse", "kind": "decode", "net": "vgg16", "n": 138344128, "K": 16, "W": 64, "density": 0.0003,
         "overwrite": False},
        # one message onto the wire and back
        {"name": "coder", "kind": "coder", "n": 25502912, "density": 0.03},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _log_int(rng, lo, hi):
    return max(int(lo), min(int(hi), int(round(_log(rng, lo, hi)))))


def _widths(rng, most):
    """2 to 5 layer widths, ordinary ones (multiples of 16) and odd ones, at most `most` weights."""
    while True:
        w = [_log_int(rng, 16, 4096) for _ in range(rng.randint(2, 5))]
        w = [v if rng.random() < 0.3 else (v + 15) // 16 * 16 for v in w]
        if rng.random() < 0.5:
            w[-1] = rng.choice([10, 100, 1000])
        sizes = [a * b for a, b in zip(w, w[1:])]
        if all(v % 4 == 0 for v in sizes[:-1]) and 2000 <= sum(sizes) <= most:      # every layer's slice is aligned
            return "-".join(str(v) for v in w)


def draw(rng):
    kind = rng.choice(["step", "host", "conv", "conv", "net", "compress", "compress", "hybrid", "decode", "decode", "coder"])
    density = round(_log(rng, 1e-4, 0.1), 6)
    if kind == "step":
        return {"kind": kind, "widths": _widths(rng, 8 << 20), "B": _log_int(rng, 8, 512), "W": _log_int(rng, 2, 64),
                "density": density, "fused": rng.random() < 0.4}
    if kind == "host":
        return {"kind": kind, "widths": _widths(rng, 2 << 20), "B": _log_int(rng, 8, 256), "density": density}
    if kind == "conv":
        while True:
            k = rng.choice([1, 1, 3, 3, 3, 5, 7])
            c = {"kind": kind, "C": _log_int(rng, 3, 1024), "H": _log_int(rng, 7, 112), "Cout": _log_int(rng, 16, 1024),
                 "k": k, "stride": rng.choice([1, 1, 2]), "pad": k // 2, "B": _log_int(rng, 4, 64),
                 "exact": rng.random() < 0.25, "accumulate": rng.random() < 0.5}
            for f in ("C", "Cout"):
                if rng.random() < 0.7 and c[f] > 4:
                    c[f] = (c[f] + 15) // 16 * 16
            if rng.random() < 0.7:
                c["H"] = rng.choice([7, 14, 28, 56, 112, 8, 16, 32, 64])
            w = work(c)
            if 2e8 <= w["flops"] <= 1e10 and w["bytes"] <= 4e8:
                return c
    if kind == "net":
        return {"kind": kind, "h": rng.choice([64, 96, 128, 160, 192, 224]), "B": _log_int(rng, 2, 30)}
    if kind == "compress":
        n = _log_int(rng, 3e4, 1.38e8)
        return {"kind": kind, "net": "", "n": n, "K": _log_int(rng, 1, min(161, n // 4096 + 1)), "density": density,
                "mask": rng.random() < 0.2}
    if kind == "hybrid":
        return {"kind": kind, "n": _log_int(rng, 3e4, 3e7), "K": 1, "W": _log_int(rng, 2, 32), "density": density / 2}
    if kind == "decode":
        n, W = _log_int(rng, 1e5, 1.38e8), _log_int(rng, 2, 64)
        return {"kind": kind, "net": "", "n": n, "K": _log_int(rng, 1, min(161, n // 4096 + 1)), "W": W,
                "density": min(density, round(2e7 / W / n, 6)), "overwrite": rng.random() < 0.5}
    return {"kind": "coder", "n": _log_int(rng, 1e5, 1.38e8), "density": min(density, 0.05)}


# ---------------------------------------------------------------------------------------------- inputs
def _uniform(n, seed):
    return torch.empty(n, device=DEV).uniform_(generator=torch.Generator(DEV).manual_seed(seed))


def _dense_layers(case):
    w = [int(v) for v in case["widths"].split("-")]
    return [wl.LayerSpec(f"fc{i}", "fc", a, b) for i, (a, b) in enumerate(zip(w, w[1:]))]


def _offsets(case):
    """Borders of the weight tensors: a network's own, or cuts whose sizes spread over orders of magnitude."""
    if case.get("net"):
        return wl.group_offsets({"resnet50": wl.resnet50_layers, "vgg16": wl.vgg16_layers}[case["net"]]())
    n, K = case["n"], case["K"]
    sizes = np.exp(np.random.RandomState(K).uniform(0, 7, K))
    cuts = np.floor(np.cumsum(sizes) / sizes.sum() * n).astype(np.int64)
    cuts[-1] = n
    return np.concatenate([[0], cuts]).astype(np.uint32)


def _ws(nbytes):
    return torch.zeros(max(int(nbytes), 256), dtype=torch.uint8, device=DEV)


def _running_state(n, offsets, density, seed):
    """g, s, r, v of a buffer whose parameters are sent every T steps, T log-normal with E[1/T] = density, each at a
    random point of its period."""
    scale = torch.pow(2.0, -20 + 8 * _uniform(len(offsets) - 1, seed))
    counts = torch.from_numpy(np.diff(offsets.astype(np.int64))).to(DEV)
    gen = torch.Generator(DEV).manual_seed(seed + 1)
    g = torch.empty(n, device=DEV).normal_(generator=gen)
    g *= torch.repeat_interleave(scale, counts, output_size=n)
    T = torch.empty(n, device=DEV).normal_(generator=gen)
    T.mul_(0.8).add_(0.32).exp_().div_(density).clamp_(min=1.0)
    decay = 1.0 - torch.exp(T * math.log(ZETA))
    s = g.square() * T.square() * ((1.0 - ZETA) / ALPHA) / decay         # r^2 = (T g)^2 meets alpha v at step T
    j = torch.floor(T.mul_(_uniform(n, seed + 2)))
    r = j * g
    v = s * ((1.0 - torch.exp(j * math.log(ZETA))) / (1.0 - ZETA))
    return g, s, r, v


def _dense_state(specs, B, density, seed):
    """x, delta of every layer, g and a running r, v whose send tests are all decided by a clear margin (the squared
    sums may differ in the last bits between correct implementations, the message may not)."""
    xs, ds, parts = [], [], []
    for i, sp in enumerate(specs):
        x, d = wl.relu_normal(sp.x_shape(B), 1.0, seed + 8 + 2 * i, DEV), wl.normal(sp.delta_shape(B), 1e-3, seed + 9 + 2 * i, DEV)
        xs.append(x)
        ds.append(d)
        parts.append((d.square().t() @ x.square()).div_(float(B) * B).reshape(-1))
    s = torch.cat(parts)
    n = s.numel()
    pick, f, u = _uniform(n, seed), _uniform(n, seed + 1), _uniform(n, seed + 2)
    q = density
    j = torch.zeros(n, device=DEV)
    f2 = f * 1e-6                                                          # never sent
    lo = 0.0
    for share, period, a, b in ((q / 3, 1, 1.5, 2.5), (q, 3, 0.37, 0.46), (7 * q / 3, 7, 0.147, 0.162)):
        here = (pick >= lo) & (pick < lo + share)                          # sent every `period` steps
        lo += share
        f2 = torch.where(here, a + (b - a) * f, f2)
        j = torch.where(here, torch.floor(u * period), j)
    sign = torch.where(_uniform(n, seed + 3) < 0.5, -1.0, 1.0)
    g = sign * (ALPHA * s * f2).sqrt()
    return xs, ds, g, j * g, j * s


def _top_exponents(g, offsets):
    """floor(log2) of each tensor's largest |g|, as another worker's message would carry (about)."""
    return torch.stack([torch.frexp(g[a:b].abs().max() + 1e-30)[1] - 1 for a, b in zip(offsets[:-1].tolist(), offsets[1:].tolist())])


def _message(n, offsets, density, seed, exps=None):
    words, gexp = wl.random_message(n, offsets, density, seed, DEV, exp_seed=11)
    if exps is not None:
        gexp = exps.to(torch.int32) + (gexp & 1)
    return words, torch.tensor([words.numel()], dtype=torch.int32, device=DEV), gexp


def _gathered(messages):
    """The W messages as an allgatherv leaves them: rows of one buffer, each with its own count."""
    L = max(4, max((m[0].numel() + 3) // 4 * 4 for m in messages))
    words = torch.zeros(len(messages), L, dtype=torch.int32, device=DEV)
    for w, m in enumerate(messages):
        words[w, :m[0].numel()] = m[0]
    counts, exps = torch.cat([m[1] for m in messages]), torch.stack([m[2] for m in messages])
    return [(words[w], counts[w:w + 1], exps[w]) for w in range(len(messages))]


def _buffers(capacity, K, n=0, mask=False):
    out = vgc.MessageBuffers(capacity, K, n, mask)
    out.words.zero_()
    return out


def _geometry(sp):
    return (sp.cin, sp.hin, sp.hin, sp.cout, sp.k, sp.k, sp.stride, sp.stride, sp.pad, sp.pad)


# ---------------------------------------------------------------------------------------------- what a program holds
def prepare(case, seed):
    kind, seed = case["kind"], int(seed) * 64
    st = {"case": case, "status": torch.zeros(1, dtype=torch.int32, device=DEV)}
    if kind in ("step", "host"):
        specs, B = _dense_layers(case), case["B"]
        offsets = wl.group_offsets(specs)
        xs, ds, g, r, v = _dense_state(specs, B, case["density"], seed)
        n, K = int(offsets[-1]), len(specs)
        s = torch.zeros(n, device=DEV)
        st.update(n=n, offsets=vgc.offsets_tensor(offsets), g=g, r=r, v=v, s=s, scale=1.0 / (float(B) * B),
                  out=_buffers(n, K), ws_c=_ws(vgc.vgc_compress_workspace_bytes(n, K)),
                  ws=_ws(max(vgc.vgc_sqgrad_linear_workspace_bytes(B, l.cin, l.cout) for l in specs)))
        if kind == "step":
            into = v if case["fused"] else s
            st["layers"] = [(x, d, into[a:b]) for x, d, a, b in zip(xs, ds, offsets[:-1].tolist(), offsets[1:].tolist())]
            exps = _top_exponents(g, offsets)
            st["others"] = _gathered([_message(n, offsets, case["density"], seed + 30 + w, exps) for w in range(case["W"] - 1)])
            st["u"] = torch.empty(n, device=DEV)
        else:
            pin = lambda t: t.cpu().pin_memory()  # noqa: E731
            st["layers"] = [{"is_conv": 0, "B": B, "C": l.cin, "Cout": l.cout, "x_host": pin(x), "delta_host": pin(d),
                             "x_dev": torch.empty_like(x), "delta_dev": torch.empty_like(d)} for l, x, d in zip(specs, xs, ds)]
            st.update(g_host=pin(g), g_dev=torch.empty_like(g), words_host=torch.zeros(n, dtype=torch.int32).pin_memory(),
                      counters_host=torch.zeros(4, dtype=torch.int32).pin_memory())
    elif kind == "conv":
        sp = _conv_spec(case)
        exact = case["exact"]
        x, d = wl.half_normal(sp.x_shape(case["B"]), 1.0, seed, DEV), wl.normal(sp.delta_shape(case["B"]), 1e-4, seed + 1, DEV)
        need = (vgc.vgc_sqgrad_conv_exact_workspace_bytes if exact else vgc.vgc_sqgrad_conv_workspace_bytes)(case["B"], *_geometry(sp))
        st.update(x=x, delta=d, S=torch.zeros(sp.n_params, device=DEV), ws=_ws(need), spec=sp, scale=1.0 / case["B"] ** 2)
    elif kind == "net":
        specs, B = wl.resnet50_layers(case["h"]), case["B"]
        offsets = wl.group_offsets(specs).tolist()
        s = torch.zeros(offsets[-1], device=DEV)
        calls, need = {}, 0
        for i, sp in enumerate(specs):
            x = wl.half_normal(sp.x_shape(B), 1.0, seed * 2 + 2 * i, DEV)
            d = wl.normal(sp.delta_shape(B), 1e-4, seed * 2 + 2 * i + 1, DEV)
            xs, ds, Ss = calls.setdefault((sp.kind, _geometry(sp)), (sp, [], [], []))[1:]
            xs.append(x)
            ds.append(d)
            Ss.append(s[offsets[i]:offsets[i + 1]])
        for sp, xs, _, _ in calls.values():
            need = max(need, vgc.vgc_sqgrad_linear_workspace_bytes(B, sp.cin, sp.cout) if sp.kind == "fc"
                       else vgc.vgc_sqgrad_conv_batch_workspace_bytes(len(xs), B, *_geometry(sp)))
        st.update(calls=list(calls.values()), s=s, ws=_ws(need), scale=1.0 / B ** 2)
    elif kind == "compress":
        offsets = _offsets(case)
        n, K = case["n"], len(offsets) - 1
        g, s, r, v = _running_state(n, offsets, case["density"], seed)
        st.update(g=g, s=s, r=r, v=v, offsets=vgc.offsets_tensor(offsets), out=_buffers(max(1024, n // 2), K, n, case["mask"]),
                  ws=_ws(vgc.vgc_compress_workspace_bytes(n, K)))
    elif kind == "hybrid":
        n, offsets = case["n"], _offsets(case)
        # a parameter is sent about every tau / |g| steps; for the larger g the variance criterion delays it further
        g = wl.normal((n,), 1e-4, seed, DEV)
        tau = float(g.abs().mean()) / case["density"]
        phase = _uniform(n, seed + 1)
        steps = (tau / g.abs().clamp_min_(1e-30)).clamp_(max=1.0 / (1.0 - ZETA))
        s = g.square() / (1.5 * ALPHA * case["density"])
        r, v = phase * tau * g.sign(), phase * steps * s
        out = vgc.HybridMessageBuffers(n, n)
        out.words.zero_()
        others = [_message(n, offsets, case["density"], seed + 8 + w) for w in range(case["W"] - 1)]
        for m in others:
            m[0].bitwise_and_(-8)                                            # sign only
        st.update(g=g, s=s, r=r, v=v, tau=tau, out=out, ws=_ws(vgc.vgc_compress_hybrid_workspace_bytes(n)),
                  others=[m[:2] for m in _gathered(others)], u=torch.empty(n, device=DEV))
    elif kind == "decode":
        n, offsets = case["n"], _offsets(case)
        st.update(messages=_gathered([_message(n, offsets, case["density"], seed + w) for w in range(case["W"])]),
                  offsets=vgc.offsets_tensor(offsets), u=wl.normal((n,), 1e-6, seed + 64, DEV))
    else:
        n = case["n"]
        words, nnz, _ = _message(n, np.array([0, n], np.uint32), case["density"], seed)
        room = torch.zeros(int(n * case["density"] * 1.25) // 4 * 4 + 1024, dtype=torch.int32, device=DEV)
        room[:words.numel()] = words
        st.update(words=room, nnz=nnz, packed=torch.zeros(vgc.vgc_pack_bound_bytes(room.numel()), dtype=torch.uint8, device=DEV),
                  packed_bytes=torch.zeros(1, dtype=torch.int32, device=DEV), back=torch.zeros_like(room),
                  ws=_ws(vgc.vgc_pack_workspace_bytes(room.numel())))
    return st


def _conv_spec(case):
    return wl.LayerSpec("conv", "conv", case["C"], case["Cout"], case["k"], case["stride"], case["pad"], case["H"])


# ---------------------------------------------------------------------------------------------- one pass
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "step":
        for x, d, S in st["layers"]:
            vgc.vgc_sqgrad_linear(x, d, st["scale"], S, case["fused"], st["ws"])
        out = vgc.vgc_compress(st["g"], None if case["fused"] else st["s"], st["r"], st["v"], st["offsets"], ALPHA, ZETA,
                               st["out"], st["ws_c"])
        vgc.vgc_decode_sum([out] + st["others"], st["offsets"], 1.0 / case["W"], st["u"], st["status"])
        return {"words": out.words, "group_exp": out.group_exp, "counters": out.counters, "r": st["r"], "v": st["v"],
                "s": st["s"], "u": st["u"], "status": st["status"]}
    if kind == "host":
        got = vgc.vgc_step_host(st["layers"], st["g_host"], st["g_dev"], st["s"], st["r"], st["v"], st["offsets"], ALPHA, ZETA,
                                st["scale"], st["out"], st["words_host"], st["counters_host"], st["ws"], st["ws_c"])
        return {"counters": list(got), "words": st["words_host"], "group_exp": st["out"].group_exp, "r": st["r"], "v": st["v"],
                "s": st["s"]}
    if kind == "conv":
        fn, sp = vgc.vgc_sqgrad_conv_exact if case["exact"] else vgc.vgc_sqgrad_conv, st["spec"]
        return fn(st["x"], st["delta"], (sp.k, sp.k), (sp.stride, sp.stride), (sp.pad, sp.pad), st["scale"], st["S"],
                  case["accumulate"], st["ws"])
    if kind == "net":
        for sp, xs, ds, Ss in st["calls"]:
            if sp.kind == "fc":
                vgc.vgc_sqgrad_linear(xs[0], ds[0], st["scale"], Ss[0], ws=st["ws"])
            else:
                vgc.vgc_sqgrad_conv_batch(xs, ds, (sp.k, sp.k), (sp.stride, sp.stride), (sp.pad, sp.pad), st["scale"], Ss,
                                          ws=st["ws"])
        return st["s"]
    if kind == "compress":
        out = vgc.vgc_compress(st["g"], st["s"], st["r"], st["v"], st["offsets"], ALPHA, ZETA, st["out"], st["ws"])
        return {"words": out.words, "group_exp": out.group_exp, "counters": out.counters, "mask": out.mask, "r": st["r"],
                "v": st["v"]}
    if kind == "hybrid":
        out = vgc.vgc_compress_hybrid(st["g"], st["s"], st["r"], st["v"], ALPHA, ZETA, st["tau"], st["out"], st["ws"])
        vgc.vgc_decode_sum_hybrid([out] + st["others"], st["tau"], 1.0 / case["W"], st["u"], st["status"])
        return {"words": out.words, "counters": out.counters, "r": st["r"], "v": st["v"], "u": st["u"], "status": st["status"]}
    if kind == "decode":
        vgc.vgc_decode_accumulate(st["messages"], st["offsets"], 1.0 / case["W"], st["u"], st["status"], overwrite=case["overwrite"])
        return {"u": st["u"], "status": st["status"]}
    vgc.vgc_pack_indices(st["words"], st["nnz"], st["packed"], st["packed_bytes"], st["status"], st["ws"])
    vgc.vgc_unpack_indices(st["packed"], st["nnz"], st["back"], st["status"])
    return {"packed": st["packed"], "packed_bytes": st["packed_bytes"], "back": st["back"], "status": st["status"]}


# ---------------------------------------------------------------------------------------------- what a pass needs
def _layer_work(sp, B, accumulate=False):
    m, n, k = sp.gemm_mnk(B)
    size = math.prod(sp.x_shape(B)) + math.prod(sp.delta_shape(B)) + m * n * (2 if accumulate else 1)
    return 4.0 * size, 2.0 * m * n * k


def _decode_bytes(n, words, overwrite):
    # an update that is written needs every element; one that is added needs the elements words point at
    return 4.0 * words + (4.0 * n if overwrite else 8.0 * min(n, words))


def work(case):
    kind = case["kind"]
    if kind in ("step", "host"):
        specs = _dense_layers(case)
        n, q = sum(l.n_params for l in specs), case["density"]
        parts = [_layer_work(l, case["B"], case.get("fused", False)) for l in specs]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
        b += n * (20 if case.get("fused") else 24) + 4.0 * n * q
        if kind == "step":
            b += _decode_bytes(n, case["W"] * n * q, True)
        else:       # over PCIe: g and the layers' tensors in, the words out
            b += sum(4.0 * case["B"] * (l.cin + l.cout) for l in specs) + 4.0 * n + 4.0 * n * q
        return {"bytes": b, "flops": f}
    if kind == "conv":
        b, f = _layer_work(_conv_spec(case), case["B"], case["accumulate"])
        return {"bytes": b, "flops": f}
    if kind == "net":
        parts = [_layer_work(l, case["B"]) for l in wl.resnet50_layers(case["h"])]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    n, q = case["n"], case["density"]
    if kind == "compress":
        return {"bytes": n * (24.0 + case["mask"]) + 4.0 * n * q, "flops": 0}
    if kind == "hybrid":
        return {"bytes": 24.0 * n + 4.0 * n * q + _decode_bytes(n, case["W"] * n * q, True), "flops": 0}
    if kind == "decode":
        return {"bytes": _decode_bytes(n, case["W"] * n * q, case["overwrite"]), "flops": 0}
    coded = max(1.0, math.ceil((math.log2(16.0 / q)) / 7.0))                # bytes of an average gap
    return {"bytes": n * q * (8.0 + 2.0 * coded), "flops": 0}


def tolerance(case):
    """The compressor and the coder are exact.  Squared sums: three tf32 products per product and fp32 sums in any order.
    Decoded updates: fp32 sums of W addends in any order."""
    kind = case["kind"]
    if kind in ("compress", "coder"):
        return "exact"
    if kind in ("hybrid", "decode"):
        return {"rel": 1e-6}
    return {"rel": 1e-5}
