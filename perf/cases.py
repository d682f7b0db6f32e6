"""Performance cases of the quantization path: what a pipeline stage asks of this library.

A stage of the pipeline receives a packed activation, unpacks and dequantizes it, and quantizes and
packs its own output for the next stage.  The cases cover the sender and the receiver, per tensor,
per channel and per token, in fp32 and bf16, with the directed search (the policy at 4 bits and
below) and with the closed-form clip, from one image to 1 GiB, on device and on host buffers.

Tensors are [images * tokens, channels] activations: x = mu_c + s_c * Laplace(0, 1) with a location
and a scale per channel, optionally 1 % outlier channels of 20 times the scale; `flat` tensors are
i.i.d. Laplace(0, 1).  A program keeps its context and its output buffers from call to call, so
they are made by prepare().
"""
from __future__ import annotations

import math

import torch

import paper_2211_04515_b200 as qp

_METHODS = {"aciq": qp.QP_CLIP_ACIQ, "search": qp.QP_CLIP_DSACIQ, "minmax": qp.QP_CLIP_MINMAX}
_DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
_CLIP = 5.0            # clip range of a received stream, in units of the Laplace scale

_context = None


def _ctx() -> qp.Context:
    """One context for the whole program, as a stage keeps it."""
    global _context
    if _context is None:
        _context = qp.Context(0)
    return _context


def _case(name, kind, rows, channels, dtype, bits, method="aciq", data="vit"):
    return {"name": name, "kind": kind, "rows": rows, "channels": channels, "dtype": dtype, "bits": bits,
            "method": method, "data": data}


def listed():
    return [
        # a latency-bound stage: one image of ViT-Base at the width of a slow link, search on
        _case("sender_1image_2bit_search", "sender", 197, 768, "f32", 2, "search"),
        # the same activation on a fast link: closed-form clip, 8 bits
        _case("sender_1image_8bit", "sender", 197, 768, "f32", 8),
        # the paper's micro-batch of 64 images, ViT-Base, search on
        _case("sender_64images_4bit_search", "sender", 64 * 197, 768, "f32", 4, "search"),
        # ViT-Huge, 128 images: larger than L2, the benchmark's workload on a slow link
        _case("sender_128images_2bit_search", "sender", 128 * 197, 1280, "f32", 2, "search"),
        # a mixed-precision stage with a ragged batch: odd row, channel and element counts
        _case("sender_ragged_bf16_6bit", "sender", 61 * 577, 769, "bf16", 6),
        # the largest tensor of the roofline sweep
        _case("sender_1gib_8bit", "sender", 1 << 18, 1 << 10, "f32", 8, "aciq", "flat"),
        # receiver of one image into a bf16 stage
        _case("receiver_1image_8bit_bf16", "receiver", 197, 768, "bf16", 8),
        # receiver of the benchmark's workload
        _case("receiver_128images_4bit", "receiver", 128 * 197, 1280, "f32", 4),
        # ViT-Large with outlier channels through the separate calls: the program looks at the
        # statistics and at the search's outcome before it sends
        _case("staged_outliers_4bit_search", "staged", 64 * 197, 1024, "f32", 4, "search", "outliers"),
        # the same tensor clipped per channel, received and sent on by one stage
        _case("channels_outliers_4bit_search", "channels", 64 * 197, 1024, "f32", 4, "search", "outliers"),
        # ViT-Huge clipped per token, received and sent on by one stage
        _case("tokens_128images_8bit", "tokens", 128 * 197, 1280, "f32", 8),
        # a stage whose link works on host memory: pinned buffers in and out
        _case("host_8images_8bit", "host", 8 * 197, 768, "f32", 8),
    ]


def draw(rng):
    kind = rng.choice(("sender", "sender", "sender", "receiver", "receiver", "staged", "channels", "tokens", "host"))
    # 150 K elements (one image) up to what the kind's listed cases stand for
    most = {"sender": 10**8, "receiver": 10**8, "staged": 1 << 25, "channels": 1 << 24, "tokens": 1 << 25,
            "host": 1 << 22}[kind]
    n = math.exp(rng.uniform(math.log(1.2e5), math.log(most)))
    channels = int(round(math.exp(rng.uniform(math.log(192), math.log(1600)))))
    if rng.random() < 0.7:
        channels = channels // 64 * 64          # most models' widths; the rest are odd ones
    rows = max(16, min(int(n / channels), 60000 if kind == "channels" else 1 << 30))
    bits = rng.choice((2, 3, 4, 6, 8) if kind in ("channels", "tokens") else (1, 2, 3, 4, 6, 8, 16))
    method = "search" if bits <= 4 and kind != "tokens" else "aciq"
    if kind == "staged" and method != "search":
        bits, method = rng.choice((2, 3, 4)), "search"
    if kind in ("sender", "tokens") and rng.random() < 0.1:
        method = "minmax"
    c = _case("", kind, rows, channels, rng.choice(("f32", "f32", "bf16")), bits, method,
              rng.choice(("vit", "vit", "outliers")))
    del c["name"]
    return c


# ------------------------------------------------------------------------------------- inputs

def _activation(case, seed):
    """(x, mu, s): the activation [rows, channels] and its channels' locations and scales (fp64)."""
    rows, channels, data = case["rows"], case["channels"], case["data"]
    dev = torch.device("cuda", 0)
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    x = torch.empty(rows, channels, device=dev).exponential_(generator=g)
    x -= torch.empty(rows, channels, device=dev).exponential_(generator=g)      # Laplace(0, 1)
    mu = torch.zeros(channels, dtype=torch.float64, device=dev)
    s = torch.ones(channels, dtype=torch.float64, device=dev)
    if data != "flat":
        mu = 0.1 * torch.randn(channels, dtype=torch.float64, device=dev, generator=g)
        s = torch.exp(0.5 * torch.randn(channels, dtype=torch.float64, device=dev, generator=g))
        if data == "outliers":
            chosen = torch.randperm(channels, device=dev, generator=g)[:max(1, round(0.01 * channels))]
            s[chosen] *= 20.0
        x.mul_(s.float()).add_(mu.float())
    return x.to(_DTYPES[case["dtype"]]), mu, s


def _quantizers(lo, hi, bits):
    """Quantizers of the clip ranges [lo, hi] in the library's layout, one row of 24 bytes each."""
    lo, hi = lo.float(), hi.float()
    span = hi.double() - lo.double()
    q = torch.zeros(lo.numel(), 6, device=lo.device)
    levels_m1 = float((1 << bits) - 1)
    q[:, 0], q[:, 1], q[:, 2], q[:, 3] = lo, hi, (span / levels_m1).float(), (levels_m1 / span).float()
    q.view(torch.int32)[:, 4] = bits
    return q


class _State:
    pass


def prepare(case, seed):
    st, ctx = _State(), _ctx()
    kind, bits, rows, channels = case["kind"], case["bits"], case["rows"], case["channels"]
    dev = torch.device("cuda", 0)
    st.ctx, st.kind, st.bits, st.rows, st.channels = ctx, kind, bits, rows, channels
    st.n, st.method, st.dtype = rows * channels, _METHODS[case["method"]], _DTYPES[case["dtype"]]
    x, mu, s = _activation(case, seed)
    nbytes = qp.qp_packed_bytes(st.n, bits)
    received = kind in ("receiver", "channels", "tokens", "host")
    if received:                                   # the stream that the stage before sent
        if kind == "channels":
            st.q_in = _quantizers(mu - _CLIP * s, mu + _CLIP * s, bits)
            st.packed_in = ctx.qp_quantize_pack_channels(x, channels, bits, st.q_in)
        elif kind == "tokens":
            b = x.float().abs().mean(1).double()
            b = torch.exp2(torch.round(torch.log2(b) * 4) / 4)
            st.q_in = _quantizers(-_CLIP * b, _CLIP * b, bits)
            st.packed_in = ctx.qp_quantize_pack_tokens(x, channels, bits, st.q_in)
        else:
            clip = _CLIP * float(s.mean())
            st.q_in = qp.qp_make_qparams(-clip, clip, bits)[1]
            st.packed_in = ctx.qp_quantize_pack(x, bits, st.q_in)
        st.y = torch.empty(st.n, dtype=st.dtype, device=dev)
    if kind != "receiver":
        st.x = x
        count = {"channels": channels, "tokens": rows}.get(kind, 1)
        st.packed = torch.empty(nbytes, dtype=torch.uint8, device=dev)
        st.q = torch.empty(count, 6, device=dev)
        st.q_values, st.q_ints = st.q[:, :4], st.q.view(torch.int32)[:, 4:]
        if kind == "tokens":
            st.stats_work = torch.empty(rows * 80, dtype=torch.uint8, device=dev)
        if kind == "staged":
            st.stats = torch.empty(10, dtype=torch.float64, device=dev)
            st.result = torch.empty(9, dtype=torch.float64, device=dev)
            si, ri = st.stats.view(torch.int64), st.result.view(torch.int32)
            st.seen = {"counts": si[:2], "moments": st.stats[2:8], "hist": si[8:], "scales": st.result[:7],
                       "chosen": ri[14:18]}
    if kind == "host":
        st.h_x, st.h_packed_in = x.cpu().pin_memory(), st.packed_in.cpu().pin_memory()
        st.h_packed = torch.empty(nbytes, dtype=torch.uint8).pin_memory()
        st.h_y = torch.empty(st.n, dtype=st.dtype).pin_memory()
        st.h_q = torch.zeros(6).pin_memory()
        st.h_q_struct = qp.QParams.from_address(st.h_q.data_ptr())
        st.h_q_values, st.h_q_ints = st.h_q[:4], st.h_q.view(torch.int32)[4:]
    return st


def run(st):
    ctx, kind, bits = st.ctx, st.kind, st.bits
    if kind == "sender":
        ctx.qp_sender_device(st.x, bits, st.method, out_packed=st.packed, out_qp=st.q)
        return st.packed, st.q_values, st.q_ints
    if kind == "receiver":
        return ctx.qp_unpack_dequantize(st.packed_in, st.n, bits, st.q_in, out=st.y)
    if kind == "staged":
        ctx.qp_stats(st.x, out=st.stats, hist_bins=qp.QP_DEFAULT_HIST_BINS)
        ctx.qp_dsaciq_search(st.x, st.stats, bits, out_result=st.result, out_qp=st.q)
        ctx.qp_quantize_pack(st.x, bits, st.q, out=st.packed)
        return st.packed, st.q_values, st.q_ints, st.seen
    if kind == "channels":
        ctx.qp_unpack_dequantize_channels(st.packed_in, st.rows, st.channels, bits, st.q_in, out=st.y)
        ctx.qp_sender_channels_device(st.x, st.channels, bits, st.method, out_packed=st.packed, out_qp=st.q)
        return st.y, st.packed, st.q_values, st.q_ints
    if kind == "tokens":
        ctx.qp_unpack_dequantize_tokens(st.packed_in, st.rows, st.channels, bits, st.q_in, out=st.y)
        ctx.qp_sender_tokens_device(st.x, st.channels, bits, st.method, out_packed=st.packed, out_qp=st.q,
                                    stats_work=st.stats_work)
        return st.y, st.packed, st.q_values, st.q_ints
    ctx.qp_receiver_host(st.h_packed_in, st.n, bits, st.q_in, st.packed_in, st.y, st.h_y)
    ctx.qp_sender_host(st.h_x, bits, st.method, st.x, st.packed, st.h_packed, st.h_q_struct)
    return st.h_y, st.h_packed, st.h_q_values, st.h_q_ints


def work(case):
    """One read of every input and one write of every output; about ten operations per element for the
    statistics and the quantizer, ten more for the search, two for the receiver."""
    n = case["rows"] * case["channels"]
    size = 4 if case["dtype"] == "f32" else 2
    kind, packed = case["kind"], qp.qp_packed_bytes(n, case["bits"])
    count = {"channels": case["channels"], "tokens": case["rows"]}.get(kind, 1)
    one_way = n * size + packed + 24 * count
    both = kind in ("channels", "tokens", "host")
    sends = kind != "receiver"
    flops = (10 * n if sends else 0) + (10 * n if case["method"] == "search" and sends else 0) + (0 if kind in ("sender", "staged") else 2 * n)
    return {"bytes": one_way * (2 if both else 1), "flops": flops}


def tolerance(case):
    """The receiver is exact.  The sender's clip ends are fp32 roundings of fp64 sums, so they may be off
    in the last place, which moves the codes of the few elements that sit on a rounding boundary: 1e-5
    of them at 8 bits, hundreds of times as many at 16.  Where every channel has a search of its own,
    neighbouring steps tie in some of the thousand channels, and the other one may be taken (a step is
    about 1e-3 of the clip)."""
    kind = case["kind"]
    if kind == "receiver":
        return "exact"
    differ = 5e-3 if case["bits"] == 16 else 3e-4
    if kind == "channels" and case["method"] == "search":
        return {"rel": 1e-3, "max": 0.05, "differ": 1e-3}
    return {"rel": 1e-5, "differ": differ}
