"""Rounding in the search with any widths: a window's float32 sum is slid at
most 15 samples from a sum formed afresh, so neither its error on noise nor the
reach of one very large sample is larger than that of runs of 16 samples."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import paper_1107_2516_gb300 as dd  # noqa: E402
from test_search_tiles_gpu import direct, run  # noqa: E402

WIDTHS = (3, 7, 20, 50)


def sums(x, widths):
    """Every window's sum as the search forms it (a threshold below them all): [width] of [rows][t], NaN past a row's end."""
    ndm, nout = x.shape
    plan = dd.Plan(4, 150.0, -1e-6, 1e-3, [0.0] * ndm, widths, -1e6, dd.DD_F32, nout)
    cands, total = plan.search(torch.from_numpy(x).cuda(), capacity=ndm * nout * len(widths))
    plan.close()
    assert total == len(cands) == ndm * sum(nout - w + 1 for w in widths)
    out = np.full((len(widths), ndm, nout), np.nan)
    out[cands["width_idx"], cands["dm_idx"], cands["t"]] = cands["value"]
    return out


def runs_of_16(x, widths):
    """Restated: a fresh sequential float32 sum at every 16th sample, the 15 between slid one sample at a time."""
    ndm, nout = x.shape
    out = np.full((len(widths), ndm, nout), np.nan)
    at = np.arange(0, nout, 16)
    pad = np.concatenate([x, np.zeros((ndm, 16 + max(widths)), np.float32)], axis=1)
    fresh, prev = np.zeros((ndm, at.size), np.float32), 0
    for p, w in enumerate(widths):
        for j in range(prev, w):
            fresh = fresh + pad[:, at + j]
        prev, b = w, fresh.copy()
        for i in range(16):
            if i:
                b = b + (pad[:, at + i - 1 + w] - pad[:, at + i - 1])
            keep = at + i < nout - w + 1
            out[p][:, at[keep] + i] = b[:, keep]
    return out


def test_error_on_noise_is_that_of_runs_of_16():
    # no window is slid further, so the expected ratio is at most 1; the sampling error of
    # the r.m.s. over 20 000 independent runs is below 1%
    x = np.random.default_rng(5).standard_normal((16, 20011)).astype(np.float32)
    c = np.concatenate([np.zeros((16, 1)), np.cumsum(x.astype(np.float64), axis=1)], axis=1)
    got, ref = sums(x, WIDTHS), runs_of_16(x, WIDTHS)
    for p, w in enumerate(WIDTHS):
        exact = c[:, w:] - c[:, :-w]
        n = exact.shape[1]
        rms = [np.sqrt(np.mean((v[p][:, :n] - exact) ** 2)) for v in (got, ref)]
        assert rms[0] <= 1.01 * rms[1], (w, rms)


@pytest.mark.parametrize("big", [2.0 ** 26, np.inf, -np.inf])
def test_reach_of_a_large_sample(big):
    # ones with one sample so large that a sum with it loses them: windows behind it are wrong until the next fresh sum
    nout = 400
    x = np.ones((64, nout), np.float32)
    x[np.arange(64), 100 + np.arange(64)] = big
    ndm = x.shape[0]
    if np.isfinite(big):
        got = sums(x, (3, 7))
    else:
        # statistics are kept while the buffer's address stays: thresholds from finite values in it
        plan = dd.Plan(4, 150.0, -1e-6, 1e-3, [0.0] * ndm, (3, 7), -1e6, dd.DD_F32, nout)
        buf = torch.linspace(0.75, 1.25, nout, device="cuda").repeat(ndm, 1)
        plan.search(buf, capacity=ndm * nout * 2)
        buf.copy_(torch.from_numpy(x))
        cands, _ = plan.search(buf, capacity=ndm * nout * 2)
        plan.close()
        got = np.full((2, ndm, nout), np.nan)
        got[cands["width_idx"], cands["dm_idx"], cands["t"]] = cands["value"]
    for p, w in enumerate((3, 7)):
        for r in range(ndm):
            at = 100 + r
            behind = got[p][r, at + 1:nout - w + 1]
            wrong = np.nonzero(behind != w)[0]
            assert np.all(got[p][r, :at - w + 1] == w)
            assert wrong.size <= 15 and (wrong.size == 0 or wrong[-1] < 15), (w, r, wrong)


@pytest.mark.parametrize("dtype", [dd.DD_F32, dd.DD_U8])
@pytest.mark.parametrize("widths", [(65,), (1, 30, 300, 3000), (64, 128, 200), (4096,), (100, 16, 4095, 31)])
def test_wide_gaps(widths, dtype):
    # widths far above the one before start from the sums of half runs (31 or 25 samples a thread);
    # small whole numbers: every sum is exact
    for nout in (4096, 4097, 3968 + 4095, 3200 + 4096, 9000):
        x = np.random.default_rng(nout).integers(0, 40, (2, nout))
        x[1, nout - 300:] += 9
        for sigma in (1.5, -0.5):
            cands, total, (mu, sg), _ = run(x, widths, sigma, dtype)
            want = direct(x.astype(np.float64), widths, mu, sg, sigma)
            got = {(int(c["dm_idx"]), int(c["t"]), int(c["width_idx"])): c["value"] for c in cands}
            assert total == len(got) == len(want) and got == want
