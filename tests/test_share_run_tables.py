"""The tables that kernel 5's configurations run with (dd_share_run_tables, host
only): every warp of stage 1 an equal share of the rows, every partial sum formed
once, the sums of dd_share_tables."""
import numpy as np
import pytest

import oracle
import synth
import paper_1107_2516_gb300 as dd
from paper_1107_2516_gb300 import build as ddbuild
from paper_1107_2516_gb300 import dd as ddc
from test_share_tables import CASES, NPMAX, SHAPES, SPLIT, _stage1_rows


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ddbuild.build()
    dd.load()


@pytest.mark.parametrize("dtype", [dd.DD_F32, dd.DD_U8, dd.DD_F16])
@pytest.mark.parametrize("config", [9, 10, 11])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_equal_shares_of_the_rows(case, config, dtype):
    nch, fch1, foff, ts, dms, _, _ = CASES[case]
    d, _ = oracle.delays(nch, fch1, foff, ts, dms)
    d = np.asarray(d)
    t, form = ddc.dd_share_run_tables(d, foff, dtype, config), ddc.dd_share_tables(d, foff, dtype, config)
    assert (t is None) == (form is None)
    if t is None:
        return
    assert t["cs"] == 4 and not t["packed"]
    db = SHAPES[config][1]
    split = db + 4 + NPMAX * 8                           # where a record's split begins
    assert np.array_equal(t["rec"][:, :, :split], form["rec"][:, :, :split])
    assert all(np.array_equal(t[k], form[k]) for k in ("base", "rlen", "rs", "pmax", "klen"))
    for b in range(t["rec"].shape[0]):
        for s in range(t["rec"].shape[1]):
            assert np.all(_stage1_rows(t["rec"][b, s], db, SPLIT[config], 100) == 1), (b, s)


def test_configuration_12():
    wl = synth.workload("lofar_f32")
    d, _ = oracle.delays(wl.nchans, wl.fch1, wl.foff, wl.tsamp, wl.dm_list)
    d = np.asarray(d)
    for dtype, packed in ((dd.DD_F32, False), (dd.DD_U8, True)):
        t, ws = ddc.dd_share_run_tables(d, wl.foff, dtype, 12), ddc.dd_share_ws_tables(d, wl.foff, dtype)
        assert t["cs"] == 4 and t["packed"] == packed
        assert all(np.array_equal(t[k], ws[k]) for k in t)
        if not packed:
            for b in range(0, t["rec"].shape[0], 8):
                for s in range(0, t["rec"].shape[1], 32):
                    assert np.all(_stage1_rows(t["rec"][b, s], 64, SPLIT[12], 100) == 1), (b, s)


def test_buffers_that_do_not_fit():
    # one subband of long rows: the sums exist, three blocks (9), five (10) or two (11) do not fit an SM
    d = np.zeros((32, 4), np.int32)
    d[:, 3] = np.arange(32) // 16 * 12000
    for config in (9, 10, 11):
        assert ddc.dd_share_tables(d, -1.0, dd.DD_F32, config) is not None
        assert ddc.dd_share_run_tables(d, -1.0, dd.DD_F32, config) is None
    with pytest.raises(dd.DDError):
        ddc.dd_share_run_tables(d, -1.0, dd.DD_F32, 5)
