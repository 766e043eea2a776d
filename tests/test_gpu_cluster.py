"""Statistic and triggers of one tile, of several and of more than a block adds up itself, against the definition on
the host (integrate.cu): tile edges, half-widths and integrations at their limits, NaNs and infinities."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_18661_gb300 import abi, inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = abi.Context(inputs.PLAIN_64S, inputs.make_weights(inputs.PLAIN_64S.net, 1))
    yield c
    c.close()


def _stat(z, n_int):
    s = np.zeros(len(z) - n_int + 1, dtype=np.float32)
    for i in range(n_int):
        s += z[i:i + len(s)]
    return s / np.float32(n_int)


def _triggers(s, h):
    """j: s[j] > s[i] for i in [j-h, j), s[j] >= s[i] for i in (j, j+h].  Short series compare index by index; in long
    ones NaN neighbours and missing sides count as -inf."""
    n, out = len(s), []
    direct = n <= 16384 and h <= 256
    t = s if direct else np.where(np.isnan(s), -np.inf, s)
    for j in range(n):
        left, right = t[max(0, j - h):j], t[j + 1:j + h + 1]
        if not direct and h > 0:
            left = np.append(left, np.float32(-np.inf)) if j < h else left
            right = np.append(right, np.float32(-np.inf)) if j + h >= n else right
        if np.all(s[j] > left) and np.all(s[j] >= right):
            out.append(j)
    return np.array(out, dtype=np.int64)


@pytest.mark.parametrize("n_out,h,n_int", [
    (1, 0, 1), (1, 16, 4), (2, 1, 1), (1023, 16, 4), (1024, 64, 16), (1025, 64, 16), (2048, 256, 1), (2049, 257, 16),
    (3000, 1024, 1024), (3000, 1025, 4), (1500, 8, 1025), (16384, 3, 16), (16385, 256, 7), (20000, 64, 16),
])
@pytest.mark.parametrize("kind", ["noise", "ties", "nonfinite"])
def test_statistic_and_triggers(ctx, n_out, h, n_int, kind):
    rng = np.random.default_rng(n_out + h)
    z = rng.standard_normal(n_out + n_int - 1).astype(np.float32)
    if kind == "ties":
        z = np.round(z).astype(np.float32)
    if kind == "nonfinite":
        z[::701] = np.nan
        z[5::977] = np.inf
        z[9::313] = -np.inf
    with np.errstate(invalid="ignore"):
        want = _stat(z, n_int)
        trig = _triggers(want, h)
    cap = max(len(trig) - 1, 1)  # the last one does not fit
    stat, idx, n = ctx.integrate(torch.from_numpy(z).cuda(), n_int, h, trig_cap=cap)
    assert np.array_equal(stat.cpu().numpy(), want, equal_nan=True)
    assert int(n) == len(trig)
    assert np.array_equal(idx.cpu().numpy()[:len(trig)], trig[:cap])


def test_more_tiles_than_a_block_adds_up(ctx):
    n, h = 8193 * 1024 + 5, 64
    z = torch.randn(n, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    stat, idx, cnt = ctx.integrate(z, 1, h, trig_cap=1 << 18)
    pad = torch.nn.functional.pad(z, (h, h), value=float("-inf"))
    left = torch.nn.functional.max_pool1d(pad[None, None, :n + h - 1], h, 1)[0, 0][:n]
    right = torch.nn.functional.max_pool1d(pad[None, None, h + 1:], h, 1)[0, 0][:n]
    want = torch.nonzero((z > left) & (z >= right))[:, 0]
    assert torch.equal(stat, z) and int(cnt) == want.numel()
    assert torch.equal(idx[:want.numel()], want)


@pytest.mark.parametrize("n_out,h,n_int", [(1, 0, 1025), (700, 0, 1500), (1500, 8, 1025), (5000, 256, 2048), (5000, 257, 2048),
                                           (16384, 64, 1025), (16385, 64, 1025)])
def test_long_integrations(ctx, n_out, h, n_int):
    """Integrations past a tile's, with NaN and -inf in some of the statistics only: a short series keeps its rule for
    both (a NaN neighbour stops a trigger, a missing side is no condition); in a long one a whole side of NaN stops it."""
    rng = np.random.default_rng(n_out + h)
    z = rng.standard_normal(n_out + n_int - 1).astype(np.float32)
    z[min(9, n_out - 1)] = -np.inf      # the first statistics: -inf
    if n_out > 100:
        z[n_int + n_out // 2] = np.nan  # statistics from n_out / 2 + 1 on, at most n_int of them
    with np.errstate(invalid="ignore"):
        want = _stat(z, n_int)
        trig = _triggers(want, h)
    if not (n_out <= 16384 and h <= 256):
        nan = np.isnan(want)
        trig = np.array([j for j in trig if not (j >= h and nan[j - h:j].all()) and
                         not (j + h < n_out and nan[j + 1:j + h + 1].all())], dtype=np.int64)
    assert np.isfinite(want).any() or n_out == 1
    stat, idx, n = ctx.integrate(torch.from_numpy(z).cuda(), n_int, h, trig_cap=max(len(trig), 1))
    assert np.array_equal(stat.cpu().numpy(), want, equal_nan=True)
    assert int(n) == len(trig)
    assert np.array_equal(idx.cpu().numpy()[:len(trig)], trig)


@pytest.mark.parametrize("n_out,h,n_int", [(700, 256, 128), (700, 257, 127), (700, 257, 128), (3000, 1024, 128),
                                           (20000, 300, 1024)])
def test_long_integrations_beside_long_clusters(ctx, n_out, h, n_int):
    """Both sides of the rule that forms the statistic before the clustering."""
    z = np.random.default_rng(n_int + h).standard_normal(n_out + n_int - 1).astype(np.float32)
    want = _stat(z, n_int)
    trig = _triggers(want, h)
    stat, idx, n = ctx.integrate(torch.from_numpy(z).cuda(), n_int, h, trig_cap=max(len(trig), 1))
    assert np.array_equal(stat.cpu().numpy(), want)
    assert int(n) == len(trig) and np.array_equal(idx.cpu().numpy()[:len(trig)], trig)
