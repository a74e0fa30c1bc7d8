"""Kernel 5's warp-specialised shape on the GPU where its forms differ:
subbands of 4 and 8 channels, packed uint8 sums, rows that start anywhere,
ragged last DM blocks and time tiles, against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import synth  # noqa: E402
import paper_1107_2516_gb300 as dd  # noqa: E402
from test_share_ws_tables import CASES, TYPE  # noqa: E402


def run(x, off, pitch, d, m, nch, fch1, foff, ts, dms, nsamp, dtype):
    flat = np.zeros(off + nch * pitch, x.dtype)
    for c in range(nch):
        flat[off + c * pitch:off + c * pitch + nsamp] = x[c]
        flat[off + c * pitch + nsamp:off + (c + 1) * pitch] = 99
    dev = torch.from_numpy(flat.view(np.int16) if dtype == "f16" else flat).cuda()
    plan = dd.Plan(nch, fch1, foff, ts, dms, [1, 2, 4], 6.0, TYPE[dtype], nsamp)
    assert plan.maxshift == m
    plan.set_tile(12, 8)
    out = torch.full((len(dms) * plan.nsamp_out + 64,), -7, dtype=torch.int32 if dtype == "u8" else torch.float32, device="cuda")
    plan.execute(dev.data_ptr() + off * flat.itemsize, pitch, out)
    _, _ = plan.search(out, allow_overflow=True)
    mu, sg = plan.stats()
    got = out.cpu().numpy()
    plan.close()
    assert np.all(got[-64:] == -7)
    return got[:-64].reshape(len(dms), nsamp - m), mu, sg


@pytest.mark.parametrize("dtype", ["f32", "u8", "f16"])
@pytest.mark.parametrize("off,pad", [(0, None), (0, 1), (3, 5), (1, None)])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_forms_against_oracle(case, off, pad, dtype):
    nch, fch1, foff, ts, dms, nsamp, _ = CASES[case]
    al = 16 // {"f32": 4, "u8": 1, "f16": 2}[dtype]
    for n in (nsamp, nsamp + 511, nsamp + 1537):
        d, m = oracle.delays(nch, fch1, foff, ts, dms)
        pitch = n + pad if pad is not None else -(-n // al) * al
        x = synth.noise_f32(nch, n, 7 + case)
        x = synth.quantize_u8(x) if dtype == "u8" else x.astype(np.float16) if dtype == "f16" else x
        got, mu, sg = run(x, off, pitch, d, m, nch, fch1, foff, ts, dms, n, dtype)
        ref = oracle.dedisperse(x if dtype == "u8" else x.astype(np.float32), np.asarray(d), n - m)
        if dtype == "u8":
            assert np.array_equal(got, ref)
        else:
            assert np.max(np.abs(got - ref)) <= 1e-5 * nch
        assert abs(mu - ref.mean()) <= 1e-5 * max(1.0, abs(ref.mean())) and abs(sg - ref.std()) <= 1e-5 * ref.std()


def test_largest_bytes():
    # every byte 255 in every channel of an 8-channel subband plan: the largest packed sums
    nch, fch1, foff, ts, dms, nsamp, _ = CASES[2]
    d, m = oracle.delays(nch, fch1, foff, ts, dms)
    x = np.full((nch, nsamp), 255, np.uint8)
    got, mu, _ = run(x, 0, nsamp + 4, d, m, nch, fch1, foff, ts, dms, nsamp, "u8")
    assert np.all(got == 255 * nch) and mu == 255.0 * nch


@pytest.mark.parametrize("dtype", ["f32", "u8", "f16"])
@pytest.mark.parametrize("case", list(range(len(CASES))) + ["kernel 3"])
def test_launches_of_few_blocks_give_the_same_sums(case, dtype):
    # the finer shape that a plan left to itself runs, against the shape it stands for
    if case == "kernel 3":                       # more delay patterns than kernel 5 takes
        nch, fch1, foff, ts, dms, nsamp, cfg = 128, 150.0, -0.1953125, 327.68e-6, [0.1 * i for i in range(41)], 3000, 5
    else:
        (nch, fch1, foff, ts, dms, nsamp, _), cfg = CASES[case], 12
    al = 16 // {"f32": 4, "u8": 1, "f16": 2}[dtype]
    x = synth.noise_f32(nch, nsamp, 3)
    x = synth.quantize_u8(x) if dtype == "u8" else x.astype(np.float16) if dtype == "f16" else x
    pitch = -(-nsamp // al) * al
    pad = np.zeros((nch, pitch), x.dtype)
    pad[:, :nsamp] = x
    dev = torch.from_numpy(pad.view(np.int16) if dtype == "f16" else pad).cuda()
    got = []
    for forced in (False, True):
        plan = dd.Plan(nch, fch1, foff, ts, dms, [1, 2], 3.0, TYPE[dtype], nsamp)
        assert plan.kernel == (3 if case == "kernel 3" else 5)
        if forced:
            plan.set_tile(cfg, 8)
        out = torch.full((len(dms) * plan.nsamp_out + 16,), -7, dtype=torch.int32 if dtype == "u8" else torch.float32, device="cuda")
        plan.execute(dev, pitch, out)
        cands, total = plan.search(out, capacity=1 << 18)
        host, n_host = plan.process_host(pad.view(np.int16) if dtype == "f16" else pad, pitch, capacity=1 << 18)
        assert n_host == total and np.array_equal(host, cands)
        got.append((out.cpu().numpy(), plan.stats()))
        plan.close()
    assert np.array_equal(got[0][0], got[1][0]) and np.all(got[0][0][-16:] == -7)
    assert got[0][1] == pytest.approx(got[1][1], rel=1e-5, abs=1e-5)


@pytest.mark.parametrize("dtype", ["f32", "u8", "f16"])
@pytest.mark.parametrize("nch,step,kernel", [(65, 0.1, 3), (64, 0.01, 5)])
@pytest.mark.parametrize("off,pad", [(0, 1), (3, 5), (1, 7), (2, None)])
def test_rows_that_start_anywhere_on_kernel_3(off, pad, nch, step, kernel, dtype):
    # a plan by itself (few blocks: the finer shape, in kernel 5's order if that is its kernel) and
    # with a shape of kernel 3 chosen
    fch1, foff, ts, dms = 150.0, -0.39, 327.68e-6, [step * i for i in range(41)]
    d, m = oracle.delays(nch, fch1, foff, ts, dms)
    al = 16 // {"f32": 4, "u8": 1, "f16": 2}[dtype]
    for nout in (1, 127, 513, 1100):
        nsamp = nout + m
        pitch = nsamp + pad if pad is not None else -(-nsamp // al) * al
        x = synth.noise_f32(nch, nsamp, 5)
        x = synth.quantize_u8(x) if dtype == "u8" else x.astype(np.float16) if dtype == "f16" else x
        flat = np.full(off + (nch - 1) * pitch + nsamp, 99, x.dtype)     # the last row ends with its samples
        for c in range(nch):
            flat[off + c * pitch:off + c * pitch + nsamp] = x[c]
        dev = torch.from_numpy(flat.view(np.int16) if dtype == "f16" else flat).cuda()
        ref = oracle.dedisperse(x if dtype == "u8" else x.astype(np.float32), np.asarray(d), nout)
        for forced in (False, True):
            plan = dd.Plan(nch, fch1, foff, ts, dms, [1], 6.0, TYPE[dtype], nsamp)
            assert plan.kernel == kernel
            if forced:
                plan.set_tile(5, 8)
            out = torch.full((len(dms) * nout + 32,), -7, dtype=torch.int32 if dtype == "u8" else torch.float32, device="cuda")
            plan.execute(dev.data_ptr() + off * flat.itemsize, pitch, out)
            plan.search(out, allow_overflow=True)
            got = out.cpu().numpy()
            plan.close()
            assert np.all(got[-32:] == -7)
            got = got[:-32].reshape(len(dms), nout)
            assert np.array_equal(got, ref) if dtype == "u8" else np.max(np.abs(got - ref)) <= 1e-5 * nch
