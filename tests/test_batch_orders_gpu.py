"""A batch beam against its plan alone: the same bits in the configuration that the
batch reports; left to itself a floating-point plan may sum in another order, a
uint8 plan not to be told apart."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import synth  # noqa: E402
import paper_1107_2516_gb300 as dd  # noqa: E402
from test_share_ws_tables import CASES, TYPE  # noqa: E402


@pytest.mark.parametrize("per_beam", [False, True])
@pytest.mark.parametrize("dtype", ["f32", "u8", "f16"])
def test_bits_of_the_reported_configuration(dtype, per_beam):
    # subbands of 4 channels (cases 0, 1, 4) and of 8 (2, 3) in configuration 12
    plans, ins, outs, pitches, refs = [], [], [], [], []
    for nch, fch1, foff, ts, dms, nsamp, _ in CASES:
        p = dd.Plan(nch, fch1, foff, ts, dms, [1, 2], 6.0, TYPE[dtype], nsamp)
        pitch = -(-nsamp // 16) * 16
        x = synth.noise_f32(nch, nsamp, nch, pitch=pitch)
        x = synth.quantize_u8(x) if dtype == "u8" else x.astype(np.float16) if dtype == "f16" else x
        d, m = oracle.delays(nch, fch1, foff, ts, dms)
        refs.append(oracle.dedisperse(x if dtype == "u8" else x.astype(np.float32), np.asarray(d), nsamp - m))
        ins.append(torch.from_numpy(x.view(np.int16) if dtype == "f16" else x).cuda())
        outs.append(torch.zeros(len(dms) * p.nsamp_out, dtype=torch.int32 if dtype == "u8" else torch.float32, device="cuda"))
        plans.append(p)
        pitches.append(pitch)
    batch = dd.Batch(plans)
    batch.set_launch_mode(per_beam)
    batch.execute(ins, pitches, outs)
    for i, p in enumerate(plans):
        cands, n = batch.results(i, allow_overflow=True)
        alone = torch.zeros_like(outs[i])
        p.execute(ins[i], pitches[i], alone)
        if dtype == "u8":
            assert torch.equal(alone, outs[i])
        else:
            assert float((alone - outs[i]).abs().max()) <= 2e-5 * CASES[i][0]      # each within 1e-5 of the exact sum
        p.set_tile(batch.beam_config(i), 8)
        p.execute(ins[i], pitches[i], alone)
        assert torch.equal(alone, outs[i])
        assert np.max(np.abs(outs[i].cpu().numpy().reshape(refs[i].shape) - refs[i])) <= (0 if dtype == "u8" else 1e-5 * CASES[i][0])
    batch.close()
    for p in plans:
        p.close()
