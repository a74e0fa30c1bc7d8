"""What a launch runs (dd_plan_get_launch) against what the plan has selected:
the finer shape of kernel 3 for few blocks, other kernels for rows that start
anywhere, the caller's choice."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import paper_1107_2516_gb300 as dd  # noqa: E402
from test_share_ws_tables import CASES, TYPE  # noqa: E402

FINER = (3, 13, 16, 128)
WS = (5, 12, 64, 512)
AL = {"f32": 4, "u8": 16, "f16": 8}


@pytest.mark.parametrize("dtype", ["f32", "u8", "f16"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_few_blocks_of_a_kernel_5_plan(case, dtype):
    nch, fch1, foff, ts, dms, nsamp, _ = CASES[case]
    plan = dd.Plan(nch, fch1, foff, ts, dms, [1], 6.0, TYPE[dtype], nsamp)
    pitch = -(-nsamp // AL[dtype]) * AL[dtype]
    buf = torch.zeros((nch + 1) * (pitch + 16) * 4, dtype=torch.uint8, device="cuda").data_ptr()
    eb = 16 // AL[dtype]
    # float sums of 8-channel subbands (cases 2 and 3) have no finer shape
    own = WS if dtype != "u8" and case in (2, 3) else FINER
    assert plan.kernel == 5 and plan.tile[0] == 12
    assert plan.launch(buf, pitch) == own
    assert plan.launch(buf, pitch + 1) == plan.launch(buf + eb, pitch) == own
    if eb > 1:
        assert plan.launch(buf + 1, pitch) == (1, -1, 16, 512)       # not on an element
    plan.set_tile(12, 8)
    assert plan.launch(buf, pitch) == plan.launch(buf, pitch + 1) == WS
    plan.set_tile(10, 8)
    assert plan.launch(buf, pitch) == (5, 10, 32, 256) and plan.launch(buf, pitch + 1) == WS
    plan.set_kernel(1)
    assert plan.kernel == 1 and plan.launch(buf, pitch) == (1, -1, 16, 512)
    plan.set_kernel(2)
    assert plan.launch(buf, pitch)[:2] == (2, 0) and plan.launch(buf, pitch + 1)[0] == 1
    plan.set_kernel(5)
    assert plan.launch(buf, pitch) == WS
    plan.set_kernel(0)
    assert plan.launch(buf, pitch) == own
    plan.close()


def test_blocks_for_every_sm():
    # as many blocks as SMs: kernel 3's own shape; more: kernel 5's; aligned rows or not
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for nch, step, want in ((65, 0.1, (3, 5, 32, 512)), (64, 0.01, WS)):
        dms = [step * i for i in range(32)]
        p0 = dd.Plan(nch, 150.0, -0.39, 327.68e-6, dms, [1], 6.0, dd.DD_F32, 1 << 17)
        m = p0.maxshift
        p0.close()
        for tiles in (16, sms - 1, sms, sms + 1):
            nsamp = 512 * tiles + m
            plan = dd.Plan(nch, 150.0, -0.39, 327.68e-6, dms, [1], 6.0, dd.DD_F32, nsamp)
            pitch = (nsamp + 3) // 4 * 4
            x = torch.zeros(nch * (pitch + 1), device="cuda")
            if want[0] == 3 and tiles < sms:
                assert plan.launch(x, pitch) == plan.launch(x, pitch + 1) == FINER
            elif tiles > sms or want[0] == 3:
                assert plan.launch(x, pitch) == plan.launch(x, pitch + 1) == want
            plan.close()


def test_arguments():
    plan = dd.Plan(4, 150.0, -0.1, 1e-3, [0.0], [1], 6.0, dd.DD_F32, 1000)
    with pytest.raises(dd.DDError):
        plan.launch(0, 1000)
    with pytest.raises(dd.DDError):
        plan.launch(16, 999)
    plan.close()


def test_the_autotuners_choice_is_what_runs():
    # 1024 channels, 128 trials x 16384 samples of float16: 64 blocks of kernel 5's shape, which leave
    # SMs empty and are still faster than the finer shape by 8%: the tuner keeps a shape that it timed as faster
    nch, foff, ts, dms = 1024, -12.0 / 1024, 327.68e-6, [0.05 * i for i in range(128)]
    p0 = dd.Plan(nch, 150.0, foff, ts, dms, [1], 6.0, dd.DD_F16, 1 << 16)
    nsamp = 16384 + p0.maxshift
    p0.close()
    pitch = -(-nsamp // 8) * 8
    x = torch.zeros(nch * pitch, dtype=torch.float16, device="cuda")
    plan = dd.Plan(nch, 150.0, foff, ts, dms, [1], 6.0, dd.DD_F16, nsamp)
    out = torch.empty(len(dms) * plan.nsamp_out, device="cuda")
    plan.autotune(x, pitch, out)
    assert plan.launch(x, pitch)[1] == plan.tile[0] != 13
    again = dd.Plan(nch, 150.0, foff, ts, dms, [1], 6.0, dd.DD_F16, nsamp)        # starts from the cached choice
    assert again.launch(x, pitch) == plan.launch(x, pitch)
    again.close()
    plan.close()


def test_the_finer_shape_is_timed_too():
    # 26 blocks of kernel 3's shape, nearly three times slower than the finer one: the tuner keeps that, also
    # after another shape was chosen, and plans of the same shape start from it
    args = (128, 150.0, -0.1953125, 327.68e-6, [0.1 * i for i in range(64)], [1], 6.0, dd.DD_F32, 8192)
    plan = dd.Plan(*args)
    x = torch.zeros(128 * 8192, device="cuda")
    out = torch.empty(64 * plan.nsamp_out, device="cuda")
    plan.set_tile(4, 8)
    plan.autotune(x, 8192, out)
    assert plan.launch(x, 8192) == FINER and plan.kernel == 3
    again = dd.Plan(*args)
    assert again.launch(x, 8192) == FINER and again.tile == plan.tile
    again.set_tile(3, 8)
    assert again.launch(x, 8192)[1] == 3
    again.close()
    plan.close()


@pytest.mark.parametrize("dtype,nout,want", [("f32", 8192, FINER), ("f16", 8192, FINER), ("u8", 8192, FINER),
                                             ("f16", 2 * 16384, WS), ("u8", 2 * 16384, WS)])
def test_the_estimate_keeps_the_faster_wave(dtype, nout, want):
    # 1024 channels, 64 trials: 16 blocks of kernel 5's shape run 2 to 2.5 times longer than the finer
    # one, 64 blocks (here in time; 128 x 16384 timed) 8% shorter for float16 and 15% for uint8
    nch, foff, ts, dms = 1024, -12.0 / 1024, 327.68e-6, [0.05 * i for i in range(64)]
    p0 = dd.Plan(nch, 150.0, foff, ts, dms, [1], 6.0, TYPE[dtype], 1 << 17)
    nsamp = nout + p0.maxshift
    p0.close()
    plan = dd.Plan(nch, 150.0, foff, ts, dms, [1], 6.0, TYPE[dtype], nsamp)
    assert plan.launch(1 << 20, -(-nsamp // 16) * 16) == want
    plan.close()


@pytest.mark.parametrize("dtype", ["f32", "u8"])
def test_one_barrier_shapes_leave_few_blocks_to_the_finer_one(dtype):
    # delay patterns that only kernel 5's shapes of 48 or 32 trials take, up to one block per SM
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nch, foff, ts, dms = 256, -12.0 / 256, 163.84e-6, [0.05 * i for i in range(64)]
    p0 = dd.Plan(nch, 150.0, foff, ts, dms, [1], 6.0, TYPE[dtype], 1 << 17)
    m = p0.maxshift
    p0.close()
    for tiles, few in ((16, True), (sms // 2, True), (sms // 2 + 1, False)):
        nsamp = 512 * tiles + m
        plan = dd.Plan(nch, 150.0, foff, ts, dms, [1], 6.0, TYPE[dtype], nsamp)
        assert plan.tile[0] == 11
        assert plan.launch(1 << 20, -(-nsamp // 16) * 16) == (FINER if few else (5, 11, 48, 512))
        plan.close()
