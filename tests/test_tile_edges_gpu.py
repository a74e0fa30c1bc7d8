"""Sizes at the edges of what a block or a step of these kernels covers: byte
sums of kernel 3 and of the subband kernel (channels four at a time, samples
in quads), binning by 2 and 4 in one pass, staged transforms of the channeliser
(128 blocks of samples at a time).  Whole-number data: exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_1107_2516_gb300 as dd  # noqa: E402


@pytest.mark.parametrize("config", [3, 4, 5, 6])
@pytest.mark.parametrize("nch", [1, 3, 4, 5, 18, 31])
def test_byte_sums_of_kernel_3(nch, config):
    rng = np.random.default_rng(nch)
    dms = [0.7 * i for i in range(37)]
    for nout in (1, 129, 511, 1030):
        d, m = oracle.delays(nch, 150.0, -0.3, 1e-3, dms)
        nsamp = nout + m
        pitch = -(-nsamp // 16) * 16
        x = rng.integers(0, 256, (nch, pitch)).astype(np.uint8)
        x[0, :] = 255
        plan = dd.Plan(nch, 150.0, -0.3, 1e-3, dms, [1], 6.0, dd.DD_U8, nsamp)
        plan.set_tile(config, 2)
        out = torch.full((len(dms) * nout + 32,), -5, dtype=torch.int32, device="cuda")
        plan.execute(torch.from_numpy(x).cuda(), pitch, out)
        plan.search(out, allow_overflow=True)
        got = out.cpu().numpy()
        ref = oracle.dedisperse(np.ascontiguousarray(x[:, :nsamp]), np.asarray(d), nout)
        assert np.array_equal(got[:-32].reshape(len(dms), nout), ref) and np.all(got[-32:] == -5)
        assert plan.stats()[0] == pytest.approx(ref.mean(), rel=1e-12)
        plan.close()


@pytest.mark.parametrize("cs", [1, 3, 4, 6, 9])
@pytest.mark.parametrize("ndm,group", [(25, 25), (40, 7)])
def test_byte_sums_of_subbands(cs, ndm, group):
    nsub, rng = 3, np.random.default_rng(cs)
    nch, dms = nsub * cs, [0.9 * i for i in range(ndm)]
    _, d1, d2, m = oracle.subband_tables(nch, 150.0, -0.3, 1e-3, dms, group, nsub)
    _, full = oracle.delays(nch, 150.0, -0.3, 1e-3, dms)       # a plan also needs more samples than the exact delays span
    for extra in (5, 700):
        nsamp = max(m, full) + extra
        nout = nsamp - m
        pitch = -(-nsamp // 16) * 16
        x = rng.integers(0, 256, (nch, pitch)).astype(np.uint8)
        plan = dd.SubbandPlan(nch, 150.0, -0.3, 1e-3, dms, group, nsub, [1], 6.0, dd.DD_U8, nsamp)
        assert plan.nsamp_out == nout
        out = torch.empty(ndm * nout, dtype=torch.int32, device="cuda")
        plan.execute(torch.from_numpy(x).cuda(), pitch, out)
        ref = oracle.subband_dedisperse(np.ascontiguousarray(x[:, :nsamp]), d1, d2, group, nout)
        assert np.array_equal(out.cpu().numpy().reshape(ndm, nout), ref)
        plan.close()


@pytest.mark.parametrize("bins", [(2,), (4,), (2, 4), (4, 2, 2), (8, 4, 2), (3, 2)])
@pytest.mark.parametrize("extra,pad", [(0, 0), (1, 15), (2, 14), (3, 13), (5, 11), (2, 1)])
def test_binning_remainders(bins, extra, pad):
    # sums of bytes over 2, 4 or 8 are exact in float32, and so are their sums over the channels
    nch, nsub, nsamp = 6, 2, 8192 + extra
    rng = np.random.default_rng(extra)
    x = rng.integers(0, 256, (nch, nsamp + pad)).astype(np.uint8)
    passes = [(10.0 * i, 10.0 * i + 4.0, 1.0, b, 2.0) for i, b in enumerate(bins)]
    plan = dd.SurveyPlan(nch, 150.0, -0.1, 1e-3, passes, nsub, [1], 6.0, dd.DD_U8, nsamp)
    outs = [torch.empty(p[0] * p[4], device="cuda") for p in plan.passes]
    plan.execute(torch.from_numpy(x).cuda(), nsamp + pad, outs)
    for i, b in enumerate(bins):
        xb = x[:, :nsamp // b * b].reshape(nch, -1, b).astype(np.float64).sum(2) / b
        dms = plan.dm_list(i)
        _, d1, d2, m = oracle.subband_tables(nch, 150.0, -0.1, 1e-3 * b, dms, 2, nsub)
        ref = oracle.subband_dedisperse(xb.astype(np.float32), d1, d2, 2, xb.shape[1] - m)
        got = outs[i].cpu().numpy().reshape(ref.shape)
        if b == 3:
            assert np.max(np.abs(got - ref)) <= 1e-5 * nch * 256
        else:
            assert np.array_equal(got, ref)
    plan.close()


@pytest.mark.parametrize("nfft", [16, 32])
@pytest.mark.parametrize("npol", [1, 2])
def test_staged_transforms(nfft, npol):
    rng = np.random.default_rng(nfft + npol)
    for blocks in (1, 127, 128, 129, 300):
        n = nfft * blocks + 2
        v = (rng.standard_normal((npol, 3, n)) + 1j * rng.standard_normal((npol, 3, n))).astype(np.complex64)
        out = torch.full((3 * nfft, blocks + 1), -1.0, device="cuda")
        dd.dd_channelise(torch.from_numpy(v.view(np.float32)).cuda(), npol, 3, n, nfft, out, blocks + 1)
        got = out.cpu().numpy().astype(np.float64)
        ref = oracle.channelise_power(v, nfft)
        # float32 transform of log2(nfft) stages: each output within 1e-6 of the largest power, as the other lengths' test
        assert np.max(np.abs(got[:, :blocks] - ref)) <= 1e-6 * nfft * ref.max()
        assert np.all(got[:, blocks] == -1.0)
