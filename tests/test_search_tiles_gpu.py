"""The search kernels at the edges of their tiles and runs (4096 or 3200 samples
a block, 32 or 25 a thread), with few, many and almost all samples above the
threshold (more than a block's hit list holds), and the finalisation over one
and several blocks of partial statistics.  The buffers hold small whole
numbers, so every boxcar sum is exact in float32 and the candidates are those
of a direct sum, value for value."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import paper_1107_2516_gb300 as dd  # noqa: E402

WIDTHS = [(1,), (2, 1), (1, 2, 4), (8, 1, 4, 2), (1, 2, 4, 8, 16), (1, 2, 4, 8, 16, 32), (64, 32, 16, 8, 4, 2, 1),
          (3, 1, 20, 7), (17, 16, 33), (5,)]


def direct(x, widths, mu, sg, k):
    """{(row, t, width index): sum} of the sums above their threshold."""
    c = np.concatenate([np.zeros((x.shape[0], 1)), np.cumsum(x, axis=1)], axis=1)
    found = {}
    for p, w in enumerate(widths):
        b = c[:, w:] - c[:, :-w]
        for r, t in zip(*np.nonzero(b > w * mu + k * sg * math.sqrt(w))):
            found[(int(r), int(t), p)] = b[r, t]
    return found


def run(x, widths, sigma, dtype, rows=False):
    nout = x.shape[1]
    plan = dd.Plan(4, 150.0, -1e-6, 1e-3, [0.0] * x.shape[0], widths, sigma, dtype, nout)
    assert plan.nsamp_out == nout
    plan.set_search_stats(rows)
    out = torch.from_numpy(x.astype(np.int32 if dtype == dd.DD_U8 else np.float32)).cuda()
    cands, total = plan.search(out, capacity=1 << 20)
    stats, row_stats = plan.stats(), plan.row_stats() if rows else None
    plan.close()
    return cands, total, stats, row_stats


@pytest.mark.parametrize("dtype", [dd.DD_F32, dd.DD_U8])
@pytest.mark.parametrize("nout", [64, 65, 127, 3199, 3200, 3201, 3263, 4095, 4096, 4097, 4159, 8192 + 31])
@pytest.mark.parametrize("sigma", [3.0, -0.5])
def test_candidates_at_tile_edges(nout, sigma, dtype):
    rng = np.random.default_rng(nout)
    for widths in WIDTHS:
        x = rng.integers(0, 40, (3, nout))
        x[1, nout - 1] += 200                       # the last sample of a row: windows that end there
        x[2, max(0, min(nout, 4096) - 40):min(nout, 4096)] += 60
        rows = widths == (1, 2, 4)
        cands, total, (mu, sg), rst = run(x, widths, sigma, dtype, rows)
        # float32 partials: sums of a block below 2^24 are exact, its mean and squares round at 2^-24
        assert abs(mu - x.mean()) <= 2.0 ** -22 * x.mean() and abs(sg - x.std()) <= 2.0 ** -20 * x.std()
        want = {}
        for r in range(3):
            m, s = (rst[0][r], rst[1][r]) if rows else (mu, sg)
            want.update({(r, t, p): b for (_, t, p), b in direct(x[r:r + 1].astype(np.float64), widths, m, s, sigma).items()})
        got = {(int(c["dm_idx"]), int(c["t"]), int(c["width_idx"])): c for c in cands}
        assert total == len(got) == len(want) and got.keys() == want.keys()
        for key, c in got.items():
            m, s = (rst[0][key[0]], rst[1][key[0]]) if rows else (mu, sg)
            w = widths[key[2]]
            assert c["value"] == want[key]
            assert c["snr"] == np.float32((want[key] - w * m) / (s * math.sqrt(w)))


@pytest.mark.parametrize("dtype", [dd.DD_F32, dd.DD_U8])
@pytest.mark.parametrize("ndm", [511, 512, 513, 1500])
def test_statistics_over_several_blocks_of_partials(ndm, dtype):
    # one partial per 4096 samples, 512 partials per finalising block
    rng = np.random.default_rng(ndm)
    x = rng.integers(0, 1000, (ndm, 4096))
    _, _, (mu, sg), _ = run(x, (1, 2), 50.0, dtype)
    # whole numbers: the per-block float32 sums stay below 2^24, so only the deviations from a block's
    # mean round (relative 2^-24 each, and so the sum of their squares)
    tol = 1e-12 if dtype == dd.DD_U8 else 2.0 ** -22
    assert abs(mu - x.mean()) <= tol * x.mean()
    assert abs(sg - x.std()) <= tol * x.std()
