"""Whitening filters built in pairs of floats (filter.cu) against taps in float64: the whitening of one impulse per
epoch returns each epoch's taps."""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_18661_gb300 import abi, inputs  # noqa: E402

pytestmark = pytest.mark.gpu

NFFT, NBIN, EPOCH = 16384, 8193, 8192
# FP32 rounding of the whitening transforms, relative to the response's norm: u per butterfly level, forward and
# inverse (2 log2 N levels): 28 x 2^-24
RTOL = 28 * 2.0 ** -24


def _taps(psd, fs, f_hp, fir):
    f = np.arange(NBIN) * fs / NFFT
    ok = (f >= f_hp) & (psd > 0)
    a = np.zeros(NBIN)
    a[ok] = psd[ok] ** -0.5
    h = np.fft.irfft(a, NFFT)
    m = np.arange(-fir // 2, fir // 2)
    return np.sqrt(2.0 / fs) * (0.5 - 0.5 * np.cos(2 * np.pi * (m + fir // 2) / fir)) * h[m]


# one and two filters per CTA, odd counts, both sides of the switch at 152; the shortest and longest taper;
# PSDs far from 1 and with bins that have no amplitude
@pytest.mark.parametrize("n_det,n_psd,fir,f_hp,scale,holes", [
    (1, 1, 2048, 32.0, 1e-46, False), (2, 1, 2048, 32.0, 1e-46, True), (3, 1, 512, 0.0, 1.0, False),
    (2, 76, 2048, 32.0, 1e-46, False), (3, 51, 2048, 32.0, 1e-46, True), (1, 153, 2046, 1024.0, 1e-46, False),
    (1, 305, 1000, 20.0, 1e-46, False), (1, 2, 2048, 32.0, 1e30, True), (1, 2, 2, 32.0, 1e-70, False),
    (1, 3, 2048, 5000.0, 1e-46, False), (2, 80, 2048, 32.0, 1e-60, True),
])
def test_filters_match_float64_taps(n_det, n_psd, fir, f_hp, scale, holes):
    wl = dataclasses.replace(inputs.PLAIN_64S, fir_len=fir, f_highpass=f_hp)
    rng = np.random.default_rng(n_det * 1000 + n_psd)
    shape = inputs.NoiseModel().psd(np.arange(NBIN) * wl.fs / NFFT) / 1e-46
    psd = scale * shape * rng.gamma(15.0, 1 / 15.0, (n_det, n_psd, NBIN))
    if holes:
        psd[..., 700:705] = [0.0, -scale, np.inf, np.nan, scale * 1e9]
    clean = np.where(np.isfinite(psd), psd, 0.0)
    half, out_len = fir // 2, n_psd * EPOCH
    amp = np.float32(np.sqrt(scale))  # taps near 1
    x = np.zeros((n_det, out_len + 2 * half), dtype=np.float32)
    x[:, half + EPOCH // 2::EPOCH][:, :n_psd] = amp
    ctx = abi.Context(wl, inputs.make_weights(wl.net, 1))
    y = ctx.whiten(torch.from_numpy(x).cuda(), torch.from_numpy(psd).cuda(), half, out_len, epoch_len=EPOCH)
    y = y.cpu().numpy().astype(np.float64).reshape(n_det, n_psd, EPOCH)
    for d in range(n_det):
        for e in sorted({0, 1, n_psd // 2, n_psd - 1} & set(range(n_psd))):
            want = np.zeros(EPOCH)
            want[EPOCH // 2 - half:EPOCH // 2 + half] = float(amp) * _taps(clean[d, e], wl.fs, f_hp, fir)
            assert np.linalg.norm(y[d, e] - want) <= RTOL * np.linalg.norm(want), (d, e)
    ctx.close()


# filters longer than the float-pair build's, few enough that the whitening's forward transforms run beside it, and more
@pytest.mark.parametrize("n_det,n_psd,fir", [(1, 1, 2050), (2, 1, 4096), (2, 3, 4096), (1, 2, 8192), (1, 153, 4096)])
def test_long_filters_behind_the_early_whitening(n_det, n_psd, fir):
    """Strain written by the kernel just before the call; the impulse of each epoch returns its taps, call after call."""
    wl = dataclasses.replace(inputs.PLAIN_64S, fir_len=fir, f_highpass=32.0)
    rng = np.random.default_rng(fir + n_psd)
    shape = inputs.NoiseModel().psd(np.arange(NBIN) * wl.fs / NFFT) / 1e-46
    psd = 1e-46 * shape * rng.gamma(15.0, 1 / 15.0, (n_det, n_psd, NBIN))
    half, out_len = fir // 2, n_psd * EPOCH
    x = torch.zeros((n_det, out_len + 2 * half), dtype=torch.float32, device="cuda")
    at = torch.arange(n_psd, device="cuda") * EPOCH + half + EPOCH // 2
    psd_d = torch.from_numpy(psd).cuda()
    ctx = abi.Context(wl, inputs.make_weights(wl.net, 1))
    for amp in (1e-23, 2e-23, 3e-23):
        amp = np.float32(amp)
        x[:, at] = float(amp)
        y = ctx.whiten(x, psd_d, half, out_len, epoch_len=EPOCH)
        y = y.cpu().numpy().astype(np.float64).reshape(n_det, n_psd, EPOCH)
        for d in range(n_det):
            for e in sorted({0, 1, n_psd // 2, n_psd - 1} & set(range(n_psd))):
                want = np.zeros(EPOCH)
                want[EPOCH // 2 - half:EPOCH // 2 + half] = float(amp) * _taps(psd[d, e], wl.fs, 32.0, fir)
                assert np.linalg.norm(y[d, e] - want) <= RTOL * np.linalg.norm(want), (d, e)
    ctx.close()
