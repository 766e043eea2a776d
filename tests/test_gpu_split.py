"""FP32 wide networks on the tensor cores (three BF16 terms per float, net_split.cu) against the FP64 oracle,
at the sizes where tiles, units and layouts can go wrong, and against the SIMT path a context with a memory
budget keeps."""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as orc  # noqa: E402
from paper_2403_18661_gb300 import abi, inputs  # noqa: E402

pytestmark = pytest.mark.gpu

LOGIT_TOL = 1e-4  # |dz| <= 1e-4 (1 + |z|): the FP32 bound of test_gpu_parity

# groups 2 .. 32 give 2 to 64 channels a group; window lengths give one row to 8192 rows per window, whole and
# ragged units of 32 positions, and tiles that hold part of a window or many
NETS = [
    (inputs.NetSpec(stem_k=7, stem_stride=2, stem_pool=1, widths=(64, 128, 256, 512), blocks=(1, 1, 1, 1), groups=16), 3072),
    (inputs.NetSpec(stem_k=7, stem_stride=2, stem_pool=1, widths=(64, 128, 256, 512), blocks=(1, 2, 1, 1), groups=32), 1024),
    (inputs.NetSpec(stem_k=3, stem_stride=1, stem_pool=0, widths=(64,), blocks=(2,), groups=32), 8192),
    (inputs.NetSpec(stem_k=5, stem_stride=2, stem_pool=0, widths=(128, 64), blocks=(1, 1), groups=1), 160),
    (inputs.NetSpec(stem_k=1, stem_stride=1, stem_pool=1, widths=(256, 256), blocks=(1, 1), groups=8), 96),
    (inputs.NetSpec(stem_k=7, stem_stride=2, stem_pool=1, widths=(64, 64, 512, 64), blocks=(1, 1, 1, 1), groups=2), 64),
]


@pytest.mark.parametrize("case", range(len(NETS)))
@pytest.mark.parametrize("n_win", [1, 3, 17])
def test_split_network_matches_oracle(case, n_win):
    net, win_len = NETS[case]
    wl = dataclasses.replace(inputs.PLAIN_64S, net=net, win_len=win_len)
    w = inputs.make_weights(net, 11 + case)
    stride, shift = 37, 129
    y = np.random.default_rng(case).standard_normal((2, (n_win - 1) * stride + win_len + 200)).astype(np.float32)
    ctx = abi.Context(wl, w)
    yd = torch.from_numpy(y).cuda()
    ctx.profile_enable()
    z = ctx.infer_windows(yd, 3, stride, n_win, shift=shift).cpu().numpy()
    assert any(k["name"] == "conv_gemm_fp32_split_tcgen05" for k in ctx.profile_read())
    ctx.sync()
    for j in {0, n_win // 2, n_win - 1}:
        a = 3 + j * stride
        l1 = np.take(y[1], np.arange(a + shift, a + shift + win_len), mode="wrap")
        want = orc.network(net, w, np.stack([y[0, a:a + win_len], l1]).astype(np.float64))
        assert abs(z[j] - want) <= LOGIT_TOL * (1 + abs(want)), (j, z[j], want)
    ctx.close()


def test_split_long_call_and_simt_path_agree():
    """More windows than one launch sequence holds, against a budgeted context (SIMT convolutions)."""
    wl = dataclasses.replace(inputs.PLAIN_64S, net=inputs.RESNET34_NET)
    w = inputs.make_weights(wl.net, 5)
    n_win = 1027
    y = torch.randn((2, (n_win - 1) * 16 + wl.win_len), device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    got = []
    for budget in (0, 32 << 30):
        ctx = abi.Context(wl, w, hbm_budget=budget)
        got.append(ctx.infer_windows(y, 0, 16, n_win).double().cpu().numpy())
        ctx.sync()
        ctx.close()
    assert np.max(np.abs(got[0] - got[1]) / (1 + np.abs(got[1]))) <= LOGIT_TOL


@pytest.mark.parametrize("n_win", [64, 152])
def test_split_tile_widths(n_win):
    """Window counts whose layers, of every stride and kernel, take tiles of 192 (64 windows) and 224 rows (152)."""
    net, win_len = NETS[0]
    wl = dataclasses.replace(inputs.PLAIN_64S, net=net, win_len=win_len)
    w = inputs.make_weights(net, 29)
    y = np.random.default_rng(n_win).standard_normal((2, (n_win - 1) * 64 + win_len)).astype(np.float32)
    ctx = abi.Context(wl, w)
    z = ctx.infer_windows(torch.from_numpy(y).cuda(), 0, 64, n_win).cpu().numpy()
    ctx.sync()
    for j in (0, 1, n_win // 3, n_win // 2, n_win - 2, n_win - 1):
        want = orc.network(net, w, y[:, j * 64:j * 64 + win_len].astype(np.float64))
        assert abs(z[j] - want) <= LOGIT_TOL * (1 + abs(want)), (j, z[j], want)
    ctx.close()


def test_split_buffers_stay_under_4_gib():
    """The largest window and width an accepted network can have: 50 MB of activations a window, so that 1024 windows
    would take 51 GB a buffer.  The call goes in shorter sequences, and its logits are those of short calls."""
    net = inputs.NetSpec(stem_k=3, stem_stride=1, stem_pool=0, widths=(512,), blocks=(1,), groups=32)
    wl = dataclasses.replace(inputs.PLAIN_64S, net=net, win_len=16384)
    w = inputs.make_weights(net, 3)
    n_win, stride = 200, 64
    y = torch.randn((2, (n_win - 1) * stride + 16384), device="cuda", generator=torch.Generator("cuda").manual_seed(9))
    ctx = abi.Context(wl, w)
    z = ctx.infer_windows(y, 0, stride, n_win)
    ctx.sync()
    assert ctx.bytes_held <= 5 * (4 << 30) + (64 << 20)
    few = abi.Context(wl, w)
    for a in (0, 100, 197):
        assert torch.equal(few.infer_windows(y, a * stride, stride, 3), z[a:a + 3])
    few.sync()
    for c in (ctx, few):
        c.close()


def test_split_on_a_device_with_little_room():
    """Room for a fraction of a launch sequence's buffers (18 GB for this network): shorter sequences, the same logits."""
    net = inputs.NetSpec(stem_k=3, stem_stride=1, stem_pool=0, widths=(512,), blocks=(1,), groups=32)
    wl = dataclasses.replace(inputs.PLAIN_64S, net=net, win_len=16384)
    w = inputs.make_weights(net, 3)
    n_win, stride = 60, 64
    y = torch.randn((2, (n_win - 1) * stride + 16384), device="cuda", generator=torch.Generator("cuda").manual_seed(9))
    ctx = abi.Context(wl, w)
    want = ctx.infer_windows(y, 0, stride, n_win)
    ctx.sync()
    ctx.close()
    ctx = abi.Context(wl, w)
    torch.cuda.empty_cache()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - (5 << 30), dtype=torch.uint8, device="cuda")
    try:
        for _ in range(2):
            assert torch.equal(ctx.infer_windows(y, 0, stride, n_win), want)
        ctx.sync()
        assert ctx.bytes_held < 5 << 30
    finally:
        del filler
        torch.cuda.empty_cache()
    ctx.close()


def test_split_of_floats_that_round_past_the_bf16_range():
    """Finite floats above the largest BF16 number, as activations (a stem bias of 3.4e38, read by convolutions with
    weights of 2^-126) and as weights (times a channel that is zero): finite in FP32, so finite here."""
    net = inputs.NetSpec(stem_k=3, stem_stride=2, stem_pool=0, widths=(64, 64), blocks=(1, 1), groups=32)
    wl = dataclasses.replace(inputs.PLAIN_64S, net=net, win_len=256)
    big = np.float32(3.4e38)
    w = inputs.make_weights(net, 5)
    parts = np.split(w, np.cumsum([int(np.prod(s)) for _, s in inputs.weight_shapes(net)])[:-1])
    parts = [p.reshape(s).copy() for p, (_, s) in zip(parts, inputs.weight_shapes(net))]
    stem_w, gamma, beta, c1 = parts[:4]
    gamma[:4], beta[0], beta[1], beta[2:4] = 0.0, big, -1.0, 1.0
    convs = [p for p in parts if p.ndim == 3 and p.shape[1] == 64]
    for p in (convs[0], convs[2], convs[4]):  # what reads the stem's output, or its residual
        p[:, 0] = np.sign(p[:, 0]) * np.float32(2.0 ** -126)
    c1[:, 1] = np.where(np.arange(3) % 2, big, -big)
    w = np.concatenate([p.ravel() for p in parts]).astype(np.float32)
    y = np.random.default_rng(2).standard_normal((2, 400)).astype(np.float32)
    ctx = abi.Context(wl, w)
    ctx.profile_enable()
    z = ctx.infer_windows(torch.from_numpy(y).cuda(), 0, 48, 3).cpu().numpy()
    assert any(k["name"] == "conv_gemm_fp32_split_tcgen05" for k in ctx.profile_read())
    ctx.sync()
    for j in range(3):
        want = orc.network(net, w, y[:, 48 * j:48 * j + 256].astype(np.float64))
        assert np.isfinite(want) and abs(z[j] - want) <= LOGIT_TOL * (1 + abs(want)), (j, z[j], want)
    ctx.close()


def test_split_workspaces_of_a_call_serve_shorter_ones():
    """1025 windows go in two sequences of 513, 1000 in one of 1000: the second call, here inside a capture, finds its
    workspaces reserved by the first."""
    net = inputs.NetSpec(stem_k=3, stem_stride=2, stem_pool=1, widths=(64,), blocks=(1,), groups=16)
    wl = dataclasses.replace(inputs.PLAIN_64S, net=net, win_len=256)
    w = inputs.make_weights(net, 3)
    y = torch.randn((2, 1024 * 16 + 256), device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    other = abi.Context(wl, w)
    want = other.infer_windows(y, 0, 16, 1000)
    ctx = abi.Context(wl, w)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        ctx.infer_windows(y, 0, 16, 1025, stream=s)
        out = torch.zeros(1000, device="cuda")
        s.synchronize()
        held = ctx.bytes_held
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            ctx.infer_windows(y, 0, 16, 1000, out=out, stream=s)
        assert ctx.bytes_held == held
        for _ in range(2):
            out.zero_()
            graph.replay()
            s.synchronize()
            assert torch.equal(out, want)
    del graph
    for c in (ctx, other):
        c.sync()
        c.close()
