"""The Welch average's sums (pairs of floats, or FP64) against the same segments' single periodograms summed in
float64 on the host: every epoch layout's branch, run boundaries, silent segments and segments far apart in power."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_18661_gb300 import abi, inputs  # noqa: E402

pytestmark = pytest.mark.gpu

NFFT, HOP = 16384, 8192
# the density factor 1 / (K ...) and its product with |X|^2 are rounded to FP32 on both sides: 4 x 2^-24
RTOL = 4 * 2.0 ** -24


# segments an epoch averages, segments from one epoch to the next: the 64 s PSDs' tree, direct pair sums, long sums
@pytest.mark.parametrize("k_seg,seg_step", [(15, 2), (15, 1), (4, 3), (16, 16), (1, 2), (31, 2)])
@pytest.mark.parametrize("kind", ["strain", "silent", "loud"])
@pytest.mark.parametrize("n_psd", [1, 32, 45])
def test_epoch_sums_match_single_periodograms(k_seg, seg_step, kind, n_psd):
    n_seg = (n_psd - 1) * seg_step + k_seg
    n = (n_seg - 1) * HOP + NFFT
    rng = np.random.default_rng(n_seg)
    x = (1e-21 * rng.standard_normal((2, n))).astype(np.float32)
    if kind == "silent":
        x[0, :5 * HOP] = 0.0
        x[1, n // 2:n // 2 + 3 * HOP] = 0.0
    if kind == "loud":  # the last segment: 2^100 times the others in power
        x[:, -HOP:] *= np.float32(2.0 ** 50)
    wl = inputs.PLAIN_64S
    ctx = abi.Context(wl, inputs.make_weights(wl.net, 1))
    xd = torch.from_numpy(x).cuda()
    one = ctx.psd_estimate(xd, n_psd=n_seg, psd_step=HOP, psd_span=NFFT).cpu().numpy()
    got = ctx.psd_estimate(xd, n_psd=n_psd, psd_step=seg_step * HOP, psd_span=(k_seg - 1) * HOP + NFFT).cpu().numpy()
    want = np.stack([one[:, e * seg_step:e * seg_step + k_seg].mean(axis=1) for e in range(n_psd)], axis=1)
    assert np.all(np.abs(got - want) <= RTOL * want)
    ctx.close()


@pytest.mark.parametrize("k_seg,seg_step", [(15, 2), (15, 1), (4, 3), (3, 5), (16, 16), (31, 2), (20, 7)])
@pytest.mark.parametrize("kind", ["loud", "nan"])
@pytest.mark.parametrize("where", ["first", "middle"])
def test_epochs_around_an_outlying_segment(k_seg, seg_step, kind, where):
    """A segment 2^100 times the others in power, or of NaN, at the start or in the middle of a run of epochs: the epochs
    that hold it are its sums, and those before and after it have none of it."""
    n_psd = 45
    n_seg = (n_psd - 1) * seg_step + k_seg
    n = (n_seg - 1) * HOP + NFFT
    x = (1e-21 * np.random.default_rng(n_seg).standard_normal((2, n))).astype(np.float32)
    a = 0 if where == "first" else n_seg // 2 * HOP + 100
    x[:, a:a + HOP] = np.nan if kind == "nan" else x[:, a:a + HOP] * np.float32(2.0 ** 50)
    wl = inputs.PLAIN_64S
    ctx = abi.Context(wl, inputs.make_weights(wl.net, 1))
    xd = torch.from_numpy(x).cuda()
    one = ctx.psd_estimate(xd, n_psd=n_seg, psd_step=HOP, psd_span=NFFT).cpu().numpy()
    got = ctx.psd_estimate(xd, n_psd=n_psd, psd_step=seg_step * HOP, psd_span=(k_seg - 1) * HOP + NFFT).cpu().numpy()
    want = np.stack([one[:, e * seg_step:e * seg_step + k_seg].mean(axis=1) for e in range(n_psd)], axis=1)
    finite = np.isfinite(want)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert finite.any() and np.all(np.abs(got[finite] - want[finite]) <= RTOL * want[finite])
    ctx.close()


@pytest.mark.parametrize("k_seg,seg_step", [(1, 1), (15, 2), (4, 3), (31, 2)])
def test_overflowing_spectrum_is_infinite(k_seg, seg_step):
    """A tone of 5e34 in one segment: its squares, scaled to the spectrum's finite part, are past FP32's range.  The
    epochs that hold the segment are infinite, not NaN, at the bins far from the tone and from its partner in the
    half-length transform (8192 - 1000, where infinities are subtracted), and the others are as they were."""
    n_psd, hit = 12, 7
    n_seg = (n_psd - 1) * seg_step + k_seg
    n = (n_seg - 1) * HOP + NFFT
    x = (1e-21 * np.random.default_rng(n_seg).standard_normal((1, n))).astype(np.float32)
    wl = inputs.PLAIN_64S
    ctx = abi.Context(wl, inputs.make_weights(wl.net, 1))

    def psd():
        return ctx.psd_estimate(torch.from_numpy(x).cuda(), n_psd=n_psd, psd_step=seg_step * HOP,
                                psd_span=(k_seg - 1) * HOP + NFFT).cpu().numpy()[0]

    quiet = psd()
    a = hit * seg_step * HOP
    x[0, a:a + NFFT] = 5e34 * np.cos(2 * np.pi * 1000 * np.arange(NFFT) / NFFT)
    got = psd()
    # segments that share samples with the tone
    seg = [s for s in range(n_seg) if abs(s * HOP - a) < NFFT]
    for e in range(n_psd):
        own = range(e * seg_step, e * seg_step + k_seg)
        if a // HOP in own:
            assert np.all(np.isinf(got[e, 2000:7000]))
        elif not set(own) & set(seg):
            assert np.all(np.abs(got[e] - quiet[e]) <= RTOL * quiet[e])
    ctx.close()


@pytest.mark.parametrize("k_seg,seg_step", [(17, 1), (32, 5), (33, 32), (16, 2), (8, 1), (40, 40), (3, 40), (16, 33)])
@pytest.mark.parametrize("n_psd", [1, 2, 5, 33])
def test_fp64_sums_at_batch_edges(k_seg, seg_step, n_psd):
    """Layouts that sum in FP64: slides and sums that end inside a batch of 8 or 16 terms, steps that share no segment."""
    n_seg = (n_psd - 1) * seg_step + k_seg
    x = (1e-21 * np.random.default_rng(n_seg).standard_normal((1, (n_seg - 1) * HOP + NFFT))).astype(np.float32)
    wl = inputs.PLAIN_64S
    ctx = abi.Context(wl, inputs.make_weights(wl.net, 1))
    xd = torch.from_numpy(x).cuda()
    one = ctx.psd_estimate(xd, n_psd=n_seg, psd_step=HOP, psd_span=NFFT).cpu().numpy()
    got = ctx.psd_estimate(xd, n_psd=n_psd, psd_step=seg_step * HOP, psd_span=(k_seg - 1) * HOP + NFFT).cpu().numpy()
    want = np.stack([one[:, e * seg_step:e * seg_step + k_seg].mean(axis=1) for e in range(n_psd)], axis=1)
    assert np.all(np.abs(got - want) <= RTOL * want)
    ctx.close()
