"""dd_process_host around the line between one launch (no more blocks than SMs)
and parts behind their input columns: the device path's candidates on both sides."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_1107_2516_gb300 as dd  # noqa: E402

# configuration: DM trials, samples per block
SHAPES = {5: (32, 512), 6: (64, 256), 9: (32, 512), 11: (48, 512), 12: (64, 512)}


@pytest.mark.parametrize("config", SHAPES)
@pytest.mark.parametrize("dtype", ["f32", "u8"])
@pytest.mark.parametrize("more", [0, 1, 9])
def test_one_launch_or_parts(more, dtype, config):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nch, foff, ts, dms = 64, -12.0 / 64, 327.68e-6, [0.002 * i for i in range(100)]
    _, m = oracle.delays(nch, 150.0, foff, ts, dms)
    trials, samples = SHAPES[config]
    nblk = -(-len(dms) // trials)
    nout = (sms // nblk + more) * samples - 3                # ragged last tile
    nsamp = nout + m
    pitch = -(-nsamp // 16) * 16
    rng = np.random.default_rng(more)
    x = rng.integers(90, 166, (nch, pitch)).astype(np.uint8 if dtype == "u8" else np.float32)
    x[:, nout // 2:nout // 2 + 3] += 20
    x[:, nout - 5:nout] += 20                                # in the last part's columns
    plan = dd.Plan(nch, 150.0, foff, ts, dms, [1, 2, 4], 4.0, dd.DD_U8 if dtype == "u8" else dd.DD_F32, nsamp)
    plan.set_tile(config, 8)
    c1, n1 = plan.process_host(torch.from_numpy(x).pin_memory(), pitch, capacity=1 << 20)
    s1 = plan.stats()
    out = torch.empty(len(dms) * nout, dtype=torch.int32 if dtype == "u8" else torch.float32, device="cuda")
    plan.execute(torch.from_numpy(x).cuda(), pitch, out)
    c2, n2 = plan.search(out, capacity=1 << 20)
    assert n1 == n2 > 100 and np.array_equal(c1[["dm_idx", "t", "width_idx", "value"]], c2[["dm_idx", "t", "width_idx", "value"]])
    assert s1 == pytest.approx(plan.stats(), rel=1e-12)
    plan.close()
