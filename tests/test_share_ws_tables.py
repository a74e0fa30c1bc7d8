"""The tables of kernel 5's warp-specialised shape (configuration 12) and the
arithmetic it does with them, restated in numpy without a GPU: subbands of 4
or 8 channels, rows that start anywhere (copies of whole 16-byte units), and
for uint8 input partial sums of four bytes a step, kept as pairs of 16 bits.
The sums equal the oracle's, every index stays inside the buffer it addresses,
and every partial sum is formed once."""
import numpy as np
import pytest

import oracle
import synth
import paper_1107_2516_gb300 as dd
from paper_1107_2516_gb300 import build as ddbuild
from paper_1107_2516_gb300 import dd as ddc

DB, TILE, NPMAX, MAXW, PW = 64, 512, 16, 8, 8
ELEM = {"f32": 4, "u8": 1, "f16": 2}
TYPE = {"f32": dd.DD_F32, "u8": dd.DD_U8, "f16": dd.DD_F16}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ddbuild.build()
    dd.load()


def patterns(r, cs):
    plen = (cs + 6) // 4 * 4
    p = r[DB + 4:DB + 4 + NPMAX * plen].reshape(NPMAX, plen).astype(np.int64)
    n = int(np.nonzero(p[:, 0] == int(r[DB]))[0][0]) + 1
    assert np.all(np.diff(p[:n, 0]) > 0)
    return p[:n], r[DB + 4 + NPMAX * plen:].astype(np.int64)


def bytes_sum(stage, pat, cs, quads, xo):
    """Stage 1 of the uint8 form for one pattern: two words per channel, cut at
    the term's byte; sums of even and odd bytes; the fifth sum from the word behind."""
    words = stage.view("<u4").astype(np.uint64)
    ev, od, nx = (np.zeros(quads.size, np.uint64) for _ in range(3))
    mask = np.uint64(0x00ff00ff)
    for c in range(cs):
        e = int(pat[1 + c]) + xo[c]
        a = np.uint64(8 * (e & 3))
        lo, hi = words[(e >> 2) + quads], words[(e >> 2) + quads + 1]
        x = ((hi << np.uint64(32) | lo) >> a) & np.uint64(0xffffffff)
        ev += x & mask
        od += (x >> np.uint64(8)) & mask
        nx += hi >> a & np.uint64(255)
    s = [ev & 0xffff, od & 0xffff, ev >> np.uint64(16), od >> np.uint64(16), nx]
    even = np.stack([s[0] | s[1] << np.uint64(16), s[2] | s[3] << np.uint64(16)], 1)
    odd = np.stack([s[1] | s[2] << np.uint64(16), s[3] | s[4] << np.uint64(16)], 1)
    return even, odd


def emulate(flat, off, pitch, nch, nsamp, d, foff, dtype):
    """out[dm][t] from the buffer `flat` whose row c starts at off + c * pitch."""
    t = ddc.dd_share_ws_tables(d, foff, TYPE[dtype])
    if t is None:
        return None, None
    cs, rs, pmax, al = t["cs"], t["rs"], t["pmax"], 16 // ELEM[dtype]
    ndm = d.shape[0]
    shifted = off % al != 0 or pitch % al != 0
    rs2 = rs + (al if shifted else 0)
    limit = nsamp if shifted else (nsamp + al - 1) // al * al
    nout = nsamp - int(d.max())
    nblk, nsub, _ = t["rec"].shape
    ntile = -(-nout // TILE)
    out = np.zeros((nblk * DB, ntile * TILE), np.int64 if dtype == "u8" else np.float64)
    rng = np.random.default_rng(0)
    for b in range(nblk):
        for j in range(ntile):
            t0 = j * TILE
            for s in range(nsub):
                # what the copies do not write: anything
                if dtype == "u8":
                    stage = rng.integers(0, 256, cs * rs2 + 64).astype(np.uint8)
                else:
                    stage = np.full(cs * rs2, np.nan)
                xo = [0] * cs
                for c in range(cs):
                    ch = s * cs + c
                    res = (off + ch * pitch) % al if shifted else 0
                    g = t0 + int(t["base"][b, ch])
                    n = max(0, min(int(t["rlen"][b, ch]), limit - g))
                    if shifted:
                        xo[c] = c * al + res
                        if n > 0:
                            n, g = -(-(n + res) // al) * al, g - res
                    src = off + ch * pitch + g
                    assert n == 0 or (src % al == 0 and n % al == 0 and n <= rs2 and 0 <= src
                                      and src + n <= -(-flat.size // al) * al)
                    stage[c * rs2:c * rs2 + n] = np.concatenate([flat, np.zeros(al, flat.dtype)])[src:src + n]
                r = t["rec"][b, s]
                pats, split = patterns(r, cs)
                q = r[:DB].astype(np.int64)
                unit = 4 if t["packed"] else 1
                # the split's rows cover every pattern's units once
                rows = (pats[:, 0] - pats[:, 1 + cs] + 31) // 32
                assert np.array_equal(np.cumsum(rows) - rows, pats[:, 2 + cs])
                assert np.array_equal(pats[1:, 1 + cs], pats[:-1, 0]) and pats[0, 1 + cs] == 0
                assert split[0] == 0 and split[PW] == rows.sum() and np.all(np.diff(split[:PW + 1]) >= 0)
                for w in range(PW):
                    if split[w] < split[w + 1]:
                        assert split[MAXW + 1 + w] == np.searchsorted(np.cumsum(rows), split[w], side="right")
                assert unit * int(r[DB]) <= pmax
                if t["packed"]:
                    P = np.zeros(pmax, np.uint64)
                    for p in pats:
                        quads = np.arange(p[1 + cs], p[0])
                        first = [(int(p[1 + c]) + xo[c] >> 2) + quads[0] for c in range(cs)]
                        last = [(int(p[1 + c]) + xo[c] >> 2) + quads[-1] + 1 for c in range(cs)]
                        assert min(first) >= 0 and 4 * max(last) + 4 <= stage.size
                        even, odd = bytes_sum(stage, p, cs, quads, xo)
                        P[2 * quads[0]:2 * quads[-1] + 2] = even.ravel()
                        P[pmax // 2 + 2 * quads[0]:pmax // 2 + 2 * quads[-1] + 2] = odd.ravel()
                    idx = q[:, None] + np.arange(TILE // 2)[None, :]
                    assert q.min() >= 0 and idx.max() < pmax
                    v = P[idx]
                    add = np.stack([v & np.uint64(0xffff), v >> np.uint64(16)], 2).reshape(DB, TILE).astype(np.int64)
                else:
                    P = np.full(pmax, np.nan)
                    for p in pats:
                        e = np.arange(p[1 + cs], p[0])
                        acc = np.zeros(e.size)
                        for c in range(cs):
                            at = int(p[1 + c]) + xo[c] + e
                            assert at.min() >= c * rs2 and at.max() < (c + 1) * rs2
                            acc += stage[at]
                        P[e] = acc
                    idx = q[:, None] + np.arange(TILE)[None, :]
                    assert q.min() >= 0 and idx.max() < int(r[DB])
                    add = P[idx]
                out[b * DB:(b + 1) * DB, t0:t0 + TILE] += add
    return out[:ndm, :nout], cs


CASES = [
    # nchans, fch1, foff, tsamp, DMs, nsamp, channels per subband expected
    (64, 150.0, -0.0234375, 163.84e-6, [0.05 * i for i in range(100)], 1700, 4),
    (72, 150.0 - 71 * 0.0234375, 0.0234375, 163.84e-6, [0.1 * i for i in range(50)], 1301, 4),      # ascending
    (64, 620.0, -0.009765625, 102.4e-6, [0.12 * i for i in range(90)], 1100, 8),
    (40, 1400.0, -0.05, 64e-6, [1.5, 0.0, 7.25, 300.0, 2.0, 2.0, 250.5] * 10, 1333, 8),             # unsorted, repeated
    (44, 1200.0, -0.05, 81.92e-6, [0.33 * i for i in range(70)], 1213, 4),                          # no multiple of 8
]


@pytest.mark.parametrize("dtype", ["f32", "u8", "f16"])
@pytest.mark.parametrize("off,pad", [(0, None), (0, 1), (3, 5), (1, None)])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_tables_reproduce_brute_force(case, off, pad, dtype):
    nch, fch1, foff, ts, dms, nsamp, want_cs = CASES[case]
    d, m = oracle.delays(nch, fch1, foff, ts, dms)
    d = np.asarray(d)
    al = 16 // ELEM[dtype]
    pitch = nsamp + pad if pad is not None else -(-nsamp // al) * al
    x = synth.noise_f32(nch, nsamp, 31 + case)
    x = synth.quantize_u8(x) if dtype == "u8" else x.astype(np.float64)
    flat = np.zeros(off + nch * pitch, x.dtype)
    for c in range(nch):
        flat[off + c * pitch:off + c * pitch + nsamp] = x[c]
        flat[off + c * pitch + nsamp:off + (c + 1) * pitch] = 77      # samples between rows: not the beam's
    got, cs = emulate(flat, off, pitch, nch, nsamp, d, foff, dtype)
    assert cs == want_cs
    ref = oracle.dedisperse(x if dtype == "u8" else x.astype(np.float32), d, nsamp - m)
    if dtype == "u8":
        assert np.array_equal(got, ref)
    else:
        assert not np.isnan(got).any() and np.max(np.abs(got - ref)) <= 1e-9 * nch


def test_more_patterns_are_refused_as_before():
    # configuration 12 takes exactly the plans whose 4-channel tables exist
    wl = synth.workload("small_f32")
    d, _ = oracle.delays(wl.nchans, wl.fch1, wl.foff, wl.tsamp, wl.dm_list)
    for dtype in TYPE.values():
        assert ddc.dd_share_tables(np.asarray(d), wl.foff, dtype, 12) is None
        assert ddc.dd_share_ws_tables(np.asarray(d), wl.foff, dtype) is None
