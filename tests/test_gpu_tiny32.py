"""The fused FP32 16-channel network (net_tiny32.cu) against the FP64 oracle: the longest and shortest windows, threads
without positions, every group size, stems of 1 to 7 taps, and more windows than clusters."""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as orc  # noqa: E402
from paper_2403_18661_gb300 import abi, inputs  # noqa: E402

pytestmark = pytest.mark.gpu

LOGIT_TOL = 1e-4  # |dz| <= 1e-4 (1 + |z|): the FP32 bound of test_gpu_parity


@pytest.mark.parametrize("win_len,groups,stem_k,blocks", [
    (3072, 8, 3, 2), (3072, 16, 7, 1), (3040, 1, 5, 3), (1632, 4, 1, 2), (96, 2, 7, 2), (32, 8, 3, 1),
])
@pytest.mark.parametrize("n_win", [1, 2, 171])
def test_fused_fp32_network_matches_oracle(win_len, groups, stem_k, blocks, n_win):
    net = dataclasses.replace(inputs.TINY_NET, groups=groups, stem_k=stem_k, blocks=(blocks,))
    wl = dataclasses.replace(inputs.PLAIN_64S, net=net, win_len=win_len)
    w = inputs.make_weights(net, win_len + groups)
    stride, shift = 37, 129
    y = np.random.default_rng(win_len).standard_normal((2, (n_win - 1) * stride + win_len + 200)).astype(np.float32)
    ctx = abi.Context(wl, w)
    yd = torch.from_numpy(y).cuda()
    ctx.profile_enable()
    z = ctx.infer_windows(yd, 5, stride, n_win, shift=shift).cpu().numpy()
    assert [k["name"] for k in ctx.profile_read()] == ["resnet_tiny_fused_fp32"]
    ctx.sync()
    want = orc.infer_windows(net, w, y.astype(np.float64), win_len, 5, stride, n_win, shift)
    assert np.max(np.abs(z - want) / (1 + np.abs(want))) <= LOGIT_TOL
    ctx.close()
