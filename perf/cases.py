"""Performance cases of the detection path: what a user of this library runs, at the sizes they run it.

Every case goes through the public Python binding (paper_2403_18661_gb300.abi).  `listed()` gives the fixed
cases, `draw(rng)` one more from the same ranges; `prepare` makes what the caller holds before the call, `run`
is one pass, `work` what the pass cannot do without, and `exact` the same outputs in 64 bits from plain torch.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2403_18661_gb300 import abi, inputs

FS, NFFT, HOP, NBIN, FIR, WIN = 2048, 16384, 8192, 8193, 2048, 3072
EPOCH, PSD_LEN, CROP = 16384, 131072, 1024
NETS = {"tiny": inputs.TINY_NET, "resnet34": inputs.RESNET34_NET}
PRECISIONS = {"fp32": abi.AFG_FP32, "bf16": abi.AFG_BF16}
TRIG_CAP = 4096  # the binding's default
LIVETIME_S = 8.64e6  # 1 day x 100 timeslides


def listed():
    return [
        # the smallest whole call: one 64 s span, 4 windows a second (a candidate follow-up, a test shot)
        dict(name="analyze_64s_tiny_bf16", kind="analyze", net="tiny", precision="bf16", stride=512, n_win=244, epochs=0),
        # the whole call in FP32 over two minutes at 16 Hz, PSDs per 8 s epoch (the hour-long search, per piece)
        dict(name="analyze_2min_resnet34_fp32", kind="analyze", net="resnet34", precision="fp32", stride=128, n_win=1920,
             epochs=1),
        # background estimation: uneven segments x timeslides in one batch, BF16
        dict(name="timeslides_3seg_12shift", kind="batch", segments="517 1204 733", n_shift=12),
        # online serving: a session of concurrent streams from open to close, 0.25 s chunks after the PSD warm-up
        dict(name="serve_32streams_72s", kind="serve", n_streams=32, seconds=72, chunk=512),
        # the network alone over strain already whitened (re-scoring with other weights): wide net on tensor cores
        dict(name="infer_resnet34_bf16", kind="infer", net="resnet34", precision="bf16", stride=128, n_win=4001, shift=0),
        # the same in FP32, a few hundred windows with a timeslide
        dict(name="infer_resnet34_fp32", kind="infer", net="resnet34", precision="fp32", stride=128, n_win=333,
             shift=2048),
        # the small net at the online rate over one hour
        dict(name="infer_tiny_bf16", kind="infer", net="tiny", precision="bf16", stride=128, n_win=57600, shift=0),
        # the small net in FP32 (reference runs)
        dict(name="infer_tiny_fp32", kind="infer", net="tiny", precision="fp32", stride=512, n_win=3601, shift=0),
        # PSD of every 8 s epoch of 6 h of two-detector strain
        dict(name="psd_6h_epochs", kind="psd", n_det=2, n_psd=2701),
        # whitening of the same 6 h, one filter per epoch and detector
        dict(name="whiten_6h_epochs", kind="whiten", n_det=2, n_psd=2701, ragged=0),
        # 16384 Hz frame data down to 2048 Hz, 1 h of two detectors
        dict(name="resample_1h_16k", kind="resample", n_det=2, n_in=3600 * 16384, factor=8),
        # one day of logits to statistic, triggers and their false-alarm rates against a timeslide background
        dict(name="rates_1day_16hz", kind="rates", n_win=1382400, n_int=16, cluster_half=64, n_bg=930464),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["analyze", "batch", "infer", "infer", "infer", "psd", "whiten", "resample", "rates"])
    if kind == "analyze":
        if rng.random() < 0.5:
            return dict(kind=kind, net="tiny", precision=rng.choice(["bf16", "fp32"]), stride=rng.choice([128, 512]),
                        n_win=rng.randint(64, 244), epochs=0)
        net = rng.choice(["tiny", "resnet34"])
        return dict(kind=kind, net=net, precision=rng.choice(["bf16", "fp32"]), stride=rng.choice([128, 256, 512]),
                    n_win=_log_int(rng, 65, 1900), epochs=1)
    if kind == "batch":
        return dict(kind=kind, segments=" ".join(str(rng.randint(300, 1200)) for _ in range(rng.randint(1, 3))),
                    n_shift=rng.randint(2, 12))
    if kind == "infer":
        net, precision = rng.choice(["tiny", "resnet34"]), rng.choice(["fp32", "bf16"])
        hi = {"tiny": {"fp32": 14400, "bf16": 57600}, "resnet34": {"fp32": 1900, "bf16": 4000}}[net][precision]
        return dict(kind=kind, net=net, precision=precision, stride=rng.choice([1, 37, 128, 512]),
                    n_win=_log_int(rng, 1, hi), shift=rng.choice([0, 2048, 5001]))
    if kind == "psd":
        return dict(kind=kind, n_det=rng.choice([1, 2, 3]), n_psd=_log_int(rng, 1, 1800))
    if kind == "whiten":
        return dict(kind=kind, n_det=rng.choice([1, 2, 3]), n_psd=_log_int(rng, 1, 1800), ragged=rng.randint(0, 9000))
    if kind == "resample":
        return dict(kind=kind, n_det=rng.choice([1, 2, 3]), n_in=_log_int(rng, 1 << 15, 3 << 24),
                    factor=rng.choice([2, 4, 5, 8, 16]))
    return dict(kind=kind, n_win=_log_int(rng, 2000, 1_400_000), n_int=rng.choice([4, 16]),
                cluster_half=rng.choice([16, 64]), n_bg=_log_int(rng, 1000, 1_000_000))


# ------------------------------------------------------------------ what each kind of case is made of

def _workload(case):
    if case["kind"] == "serve":
        return inputs.SERVING_128
    if case["kind"] == "batch":
        return inputs.TIMESLIDE_DAY
    base = inputs.PLAIN_64S
    net = NETS[case.get("net", "tiny")]
    if case["kind"] == "analyze":
        return dataclasses.replace(base, net=net, stride=case["stride"], n_win=case["n_win"],
                                   epoch_len=EPOCH if case["epochs"] else 0)
    if case["kind"] == "whiten":
        return dataclasses.replace(base, net=net, epoch_len=EPOCH)
    return dataclasses.replace(base, net=net)


def _weights(case, seed):
    return inputs.make_weights(_workload(case).net, 77 + seed)


def _context(case, seed):
    return abi.Context(_workload(case), _weights(case, seed), precision=PRECISIONS[case.get("precision", "bf16")])


def _generator(seed, salt):
    return torch.Generator(device="cuda").manual_seed(1000003 * salt + seed)


def _shaped_noise(n_det, n, seed, salt, fs=FS, whitened=False):
    """Gaussian noise [n_det][n]: detector noise of inputs.NoiseModel, or (whitened) unit noise above 32 Hz."""
    m = 1 << (n - 1).bit_length()
    f = torch.arange(m // 2 + 1, dtype=torch.float64, device="cuda") * (fs / m)
    if whitened:
        amp = (f >= 32.0).to(torch.float64)
    else:
        mod = inputs.NoiseModel()
        u = f.clamp_min(mod.f_flat) / mod.f0
        amp = torch.sqrt(mod.S0 * (mod.a * u ** -4.14 + mod.b + mod.c * u * u) * (fs / 2.0))
    g = _generator(seed, salt)
    out = torch.empty((n_det, n), dtype=torch.float32, device="cuda")
    for d in range(n_det):
        w = torch.randn(m, dtype=torch.float64, device="cuda", generator=g)
        out[d] = torch.fft.irfft(torch.fft.rfft(w) * amp, n=m)[:n].to(torch.float32)
    return out


def _n_raw(case):
    return PSD_LEN + case["n_psd"] * EPOCH + CROP + case.get("ragged", 0)


def _whiten_span(case):
    return case["n_psd"] * EPOCH + case["ragged"]


def _infer_len(case):
    return (case["n_win"] - 1) * case["stride"] + WIN + 6000


def _segment_seconds(case):
    return [int(s) for s in case["segments"].split()]


def _segments(case):
    segs, off = [], 0
    for s in _segment_seconds(case):
        segs.append((off, s * FS))
        off += s * FS
    return segs, off


def _serve_len(case):
    return case["seconds"] * FS


def _logits(case, seed):
    """Logits as the network gives them: neighbouring windows overlap, so they are correlated."""
    w = torch.randn(case["n_win"] + 12, device="cuda", generator=_generator(seed, 5))
    return w.unfold(0, 13, 1).mean(-1).mul_(1.5)


def _background(case, seed):
    """Timeslide background: the largest of a hundred correlated draws each, so a Gumbel-like tail."""
    u = torch.rand(case["n_bg"], dtype=torch.float64, device="cuda", generator=_generator(seed, 6)).clamp_min(1e-12)
    return (0.9 - 0.12 * torch.log(-torch.log(u))).to(torch.float32)


def _make_inputs(case, seed):
    """Device tensors of one case (host arrays for serving) from the seed alone."""
    kind = case["kind"]
    if kind == "analyze":
        return dict(x=_shaped_noise(2, _workload(case).n_raw, seed, 1))
    if kind == "batch":
        return dict(x=_shaped_noise(2, _segments(case)[1], seed, 2))
    if kind == "serve":
        n = _serve_len(case)
        x = _shaped_noise(2 * case["n_streams"], n, seed, 3).view(case["n_streams"], 2, n)
        return dict(x=x.cpu().numpy())
    if kind == "infer":
        return dict(y=_shaped_noise(2, _infer_len(case), seed, 4, whitened=True))
    if kind == "psd":
        return dict(x=_shaped_noise(case["n_det"], _n_raw(case), seed, 7))
    if kind == "whiten":
        x = _shaped_noise(case["n_det"], _n_raw(case), seed, 8)
        return dict(x=x, psd=_welch64(x, case["n_psd"], EPOCH, PSD_LEN))
    if kind == "resample":
        return dict(x=_shaped_noise(case["n_det"], case["n_in"], seed, 9, fs=FS * case["factor"]))
    return dict(logits=_logits(case, seed), bg=_background(case, seed))


def prepare(case, seed):
    state = dict(case=case, ctx=_context(case, seed), **_make_inputs(case, seed))
    wl, ctx = _workload(case), state["ctx"]
    dev = dict(device="cuda")
    if case["kind"] == "analyze":
        state["out"] = (torch.empty(wl.n_win, dtype=torch.float32, **dev),
                        torch.empty(wl.n_win - wl.n_int + 1, dtype=torch.float32, **dev),
                        torch.zeros(TRIG_CAP, dtype=torch.int64, **dev), torch.zeros(1, dtype=torch.int64, **dev))
    elif case["kind"] == "batch":
        segs, _ = _segments(case)
        _, windows, stats = ctx.batch_layout(segs, case["n_shift"], FS)
        state["segs"] = segs
        state["out"] = (torch.empty(windows, dtype=torch.float32, **dev), torch.empty(stats, dtype=torch.float32, **dev),
                        torch.zeros(TRIG_CAP, dtype=torch.int64, **dev), torch.zeros(1, dtype=torch.int64, **dev))
    elif case["kind"] == "serve":
        # what the clients send, round by round: long chunks through the PSD warm-up, then the online ones
        x, bounds, pos = state.pop("x"), [], 0
        warm = PSD_LEN + CROP
        while pos < x.shape[2]:
            step = 4096 if pos + 4096 <= warm else case["chunk"]
            bounds.append((pos, min(pos + step, x.shape[2])))
            pos = bounds[-1][1]
        state["rounds"] = [np.ascontiguousarray(x[:, :, a:b]) for a, b in bounds]
        # (twice the slots: a closed stream's is free again once the engine has gone round)
        ctx.stream_start(max_streams=2 * case["n_streams"], max_chunk=4096)
    elif case["kind"] == "rates":
        state["n_bg"] = torch.tensor([case["n_bg"]], dtype=torch.int64, **dev)
    return state


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "analyze":
        return ctx.analyze(state["x"], trig_cap=TRIG_CAP, out=state["out"])
    if kind == "batch":
        return ctx.batch_run(state["x"], state["segs"], case["n_shift"], FS, trig_cap=TRIG_CAP, out=state["out"])
    if kind == "serve":
        sids = [ctx.stream_open() for _ in range(case["n_streams"])]
        for chunk in state["rounds"]:
            ctx.stream_push_many(sids, chunk)
        ctx.stream_flush()
        res = [ctx.stream_poll(s) for s in sids]
        for s in sids:
            ctx.stream_close(s)
        return [np.stack([r[k] for r in res]) for k in ("logit", "stat", "window")]
    if kind == "infer":
        return ctx.infer_windows(state["y"], 0, case["stride"], case["n_win"], shift=case["shift"])
    if kind == "psd":
        return ctx.psd_estimate(state["x"], n_psd=case["n_psd"], psd_step=EPOCH, psd_span=PSD_LEN)
    if kind == "whiten":
        return ctx.whiten(state["x"], state["psd"], PSD_LEN, _whiten_span(case), epoch_len=EPOCH)
    if kind == "resample":
        return ctx.resample(state["x"], case["factor"])[0]
    stat, trig, n_trig = ctx.integrate(state["logits"], case["n_int"], case["cluster_half"], trig_cap=TRIG_CAP)
    trig = trig[:min(int(n_trig), TRIG_CAP)]  # the caller reads how many triggers there are
    n_above, far, bg_sorted = ctx.far(state["bg"], stat[trig], LIVETIME_S, n_bg=state["n_bg"])
    return stat, trig, n_trig, n_above, far, bg_sorted


# ------------------------------------------------------------------ work

def _net_flops(net):
    length = (WIN + 2 * (net.stem_k // 2) - net.stem_k) // net.stem_stride + 1
    c = net.widths[0]
    total = 2 * length * c * net.in_ch * net.stem_k
    if net.stem_pool:
        length = (length - 1) // 2 + 1
    for s, (w, nb) in enumerate(zip(net.widths, net.blocks)):
        for b in range(nb):
            stride = 2 if s > 0 and b == 0 else 1
            out = (length - 1) // stride + 1
            total += 2 * out * w * (3 * c + 3 * w + (c if stride != 1 or c != w else 0))
            length, c = out, w
    return total


def _spectral_flops(n_seg, n_filter, n_out):
    """Welch: a real transform a segment; a filter: an inverse and a forward transform of a real, even sequence;
    whitening: a forward and an inverse real transform per 16385 - F outputs."""
    real = 2.5 * NFFT * math.log2(NFFT)
    return real * (n_seg + n_filter + 2.0 * n_out / (NFFT + 1 - FIR))


def work(case):
    kind, wl = case["kind"], _workload(case)
    w_bytes = 4 * inputs.n_weights(wl.net)
    if kind == "analyze":
        n_stat = wl.n_win - wl.n_int + 1
        n_seg = (2 * wl.n_epochs + 13) if case["epochs"] else 15
        return dict(bytes=8 * wl.n_raw + 4 * (wl.n_win + n_stat) + w_bytes,
                    flops=wl.n_win * _net_flops(wl.net) + _spectral_flops(2 * n_seg, 2 * wl.n_epochs, 2 * wl.n_white))
    if kind == "batch":
        n_ep = [(s * FS - PSD_LEN - CROP) // EPOCH for s in _segment_seconds(case)]
        n_win = sum((e * EPOCH - WIN) // wl.stride + 1 for e in n_ep) * case["n_shift"]
        return dict(bytes=8 * FS * sum(_segment_seconds(case)) + 8 * n_win + w_bytes,
                    flops=n_win * _net_flops(wl.net) + sum(_spectral_flops(2 * (2 * e + 13), 2 * e, 2 * e * EPOCH)
                                                           for e in n_ep))
    if kind == "serve":
        q = _serve_len(case) - PSD_LEN - CROP + 1
        n_win, n_ep = (q - WIN) // wl.stride + 1, -(-q // EPOCH)
        return dict(bytes=case["n_streams"] * (8 * _serve_len(case) + 16 * n_win) + w_bytes,
                    flops=case["n_streams"] * (n_win * _net_flops(wl.net) +
                                               _spectral_flops(2 * (2 * n_ep + 13), 2 * n_ep, 2 * q)))
    if kind == "infer":
        return dict(bytes=8 * _infer_len(case) + 4 * case["n_win"] + w_bytes, flops=case["n_win"] * _net_flops(wl.net))
    if kind == "psd":
        return dict(bytes=case["n_det"] * (4 * (PSD_LEN + (case["n_psd"] - 1) * EPOCH) + 8 * NBIN * case["n_psd"]),
                    flops=_spectral_flops(case["n_det"] * (2 * case["n_psd"] + 13), 0, 0))
    if kind == "whiten":
        n = _whiten_span(case)
        return dict(bytes=case["n_det"] * (4 * (2 * n + FIR - 1) + 8 * NBIN * case["n_psd"]),
                    flops=_spectral_flops(0, case["n_det"] * case["n_psd"], case["n_det"] * n))
    if kind == "resample":
        n_out = case["n_in"] // case["factor"]
        return dict(bytes=4 * case["n_det"] * (case["n_in"] + n_out),
                    flops=2 * case["n_det"] * n_out * (20 * case["factor"] + 1))
    return dict(bytes=4 * (2 * case["n_win"] + 2 * case["n_bg"]) + TRIG_CAP * (8 + 4 + 8 + 8),
                flops=case["n_win"] * 2)


# ------------------------------------------------------------------ the same in 64 bits

def _welch64(x, n_psd, step, span):
    n = torch.arange(NFFT, dtype=torch.float64, device=x.device)
    win = 0.5 - 0.5 * torch.cos(2.0 * math.pi * n / NFFT)
    k_seg = (span - NFFT) // HOP + 1
    seg_step = step // HOP if n_psd > 1 else 1
    used = ((n_psd - 1) * seg_step + k_seg - 1) * HOP + NFFT
    psd = torch.empty((x.shape[0], n_psd, NBIN), dtype=torch.float64, device=x.device)
    for d in range(x.shape[0]):
        segs = x[d, :used].unfold(0, NFFT, HOP)
        p = torch.cat([torch.fft.rfft(s.to(torch.float64) * win).abs().square() for s in segs.split(512)])
        p[:, 1:NFFT // 2] *= 2.0
        p /= FS * win.square().sum()
        psd[d] = p.unfold(0, k_seg, seg_step)[:n_psd].mean(-1)
    return psd


def _whiten64(x, psd, out_first, out_len, epoch_len):
    """The linear FIR of every epoch's taps, by zero-padded FFTs."""
    n_ep = -(-out_len // epoch_len) if epoch_len else 1
    span = epoch_len or out_len
    f = torch.arange(NBIN, dtype=torch.float64, device=x.device) * (FS / NFFT)
    m = torch.arange(-FIR // 2, FIR // 2, dtype=torch.float64, device=x.device)
    taper = math.sqrt(2.0 / FS) * (0.5 - 0.5 * torch.cos(2.0 * math.pi * (m + FIR // 2) / FIR))
    a = out_first - FIR // 2 + 1
    nf = 1 << (span + FIR - 2).bit_length()
    y = torch.empty((x.shape[0], n_ep * span), dtype=torch.float64, device=x.device)
    for d in range(x.shape[0]):
        row = x[d, a:a + out_len + FIR - 1]  # (the oldest tap is zero, so one sample past the end may be missing)
        row = torch.nn.functional.pad(row, (0, n_ep * span + FIR - 1 - row.shape[0]))
        blocks = row.unfold(0, span + FIR - 1, span)
        for lo in range(0, n_ep, 256):
            hi = min(lo + 256, n_ep)
            p = psd[d, torch.arange(lo, hi, device=x.device).clamp_max(psd.shape[1] - 1)]
            h = torch.fft.irfft(torch.where((f >= 32.0) & (p > 0), p.rsqrt(), 0.0).to(torch.complex128), n=NFFT)
            taps = torch.cat([h[:, -FIR // 2:], h[:, :FIR // 2]], 1) * taper
            c = torch.fft.irfft(torch.fft.rfft(blocks[lo:hi].to(torch.float64), n=nf) * torch.fft.rfft(taps, n=nf), n=nf)
            y[d, lo * span:hi * span] = c[:, FIR - 1:FIR - 1 + span].reshape(-1)
    return y[:, :out_len]


def _net64(net, weights, win):
    """Logits [n] of windows win [n][2][W] (float64)."""
    it = iter(torch.split(torch.from_numpy(weights.astype(np.float64)).to(win.device),
                          [int(np.prod(s)) for _, s in inputs.weight_shapes(net)]))
    shapes = iter([s for _, s in inputs.weight_shapes(net)])

    def conv_gn(x, stride):  # x [n][L][C]: convolution (padding k // 2) and GroupNorm
        w, gamma, beta = (next(it).view(next(shapes)) for _ in range(3))
        k = w.shape[2]
        xp = torch.nn.functional.pad(x, (0, 0, k // 2, k // 2))
        length = (x.shape[1] + 2 * (k // 2) - k) // stride + 1
        cols = torch.cat([xp[:, r:r + (length - 1) * stride + 1:stride] for r in range(k)], 2)
        y = cols @ w.permute(2, 1, 0).reshape(-1, w.shape[0])
        g = y.view(y.shape[0], length, net.groups, -1)
        var, mean = torch.var_mean(g, dim=(1, 3), unbiased=False, keepdim=True)
        return ((g - mean) * torch.rsqrt(var + net.eps)).view_as(y) * gamma + beta

    x = torch.relu(conv_gn(win.transpose(1, 2), net.stem_stride))
    if net.stem_pool:
        x = torch.nn.functional.max_pool1d(x.transpose(1, 2), 3, 2, 1).transpose(1, 2)
    cin = net.widths[0]
    for s, (width, nb) in enumerate(zip(net.widths, net.blocks)):
        for b in range(nb):
            stride = 2 if s > 0 and b == 0 else 1
            h = conv_gn(torch.relu(conv_gn(x, stride)), 1)
            x = torch.relu(h + (conv_gn(x, stride) if stride != 1 or cin != width else x))
            cin = width
    fc_w, fc_b = next(it), next(it)
    return x.mean(1) @ fc_w + fc_b


def _infer64(net, weights, y, stride, n_win, shift):
    y = torch.stack([y[0], torch.roll(y[1], -shift)]).to(torch.float64)
    win = y.unfold(1, WIN, stride)[:, :n_win].transpose(0, 1)
    per = 64 if net.stem_pool else 512
    return torch.cat([_net64(net, weights, w) for w in win.split(per)])


def _stat64(logits, n_int):
    return logits.unfold(0, n_int, 1).mean(-1)


def _white_epochs64(x, n_ep, out_len):
    psd = _welch64(x, n_ep, EPOCH, PSD_LEN)
    return _whiten64(x, psd, PSD_LEN, out_len, EPOCH)


def exact(case, seed):
    kind, wl = case["kind"], _workload(case)
    if kind == "rates":
        return _stat64(_logits(case, seed).to(torch.float64), case["n_int"]), None, None, None, None, None
    if kind == "resample":
        return _resample64(_make_inputs(case, seed)["x"], case["factor"])
    w, data = _weights(case, seed), _make_inputs(case, seed)
    if kind == "analyze":
        x = data["x"]
        if case["epochs"]:
            y = _white_epochs64(x, wl.n_epochs, wl.n_white)
        else:
            y = _whiten64(x, _welch64(x, 1, 0, wl.n_raw), CROP, wl.n_white, 0)
        z = _infer64(wl.net, w, y, wl.stride, wl.n_win, 0)
        return z, _stat64(z, wl.n_int), None, None
    if kind == "batch":
        logits, stats = [], []
        for off, n in _segments(case)[0]:
            n_ep = (n - PSD_LEN - CROP) // EPOCH
            y = _white_epochs64(data["x"][:, off:off + n], n_ep, n_ep * EPOCH)
            n_win = (n_ep * EPOCH - WIN) // wl.stride + 1
            for k in range(1, case["n_shift"] + 1):
                z = _infer64(wl.net, w, y, wl.stride, n_win, k * FS)
                logits.append(z)
                stats.append(_stat64(z, wl.n_int))
        return torch.cat(logits), torch.cat(stats), None, None
    if kind == "serve":
        logits, stats = [], []
        for x in torch.from_numpy(data["x"]).cuda():
            q = x.shape[1] - PSD_LEN - CROP + 1
            y = _white_epochs64(x, -(-q // EPOCH), q)
            z = _infer64(wl.net, w, y, wl.stride, (q - WIN) // wl.stride + 1, 0)
            logits.append(z[wl.n_int - 1:].cpu().numpy())
            stats.append(_stat64(z, wl.n_int).cpu().numpy())
        return [np.stack(logits), np.stack(stats), None]
    if kind == "infer":
        return _infer64(wl.net, w, data["y"], case["stride"], case["n_win"], case["shift"])
    if kind == "psd":
        return _welch64(data["x"], case["n_psd"], EPOCH, PSD_LEN)
    return _whiten64(data["x"], data["psd"], PSD_LEN, _whiten_span(case), EPOCH)


def _resample64(x, factor):
    """Kaiser-windowed sinc (beta 5), 20 factor + 1 taps, cutoff at the output Nyquist, unit gain at DC."""
    half = 10 * factor
    k = torch.arange(-half, half + 1, dtype=torch.float64, device=x.device)
    h = torch.sinc(k / factor) * torch.special.i0(5.0 * torch.sqrt((1.0 - (k / half) ** 2).clamp_min(0.0)))
    h /= h.sum()
    y = []
    for row in x:
        seg = row.unfold(0, 2 * half + 1, factor)
        y.append(torch.cat([s.to(torch.float64) @ h for s in seg.split(1 << 20)]))
    return torch.stack(y)
