"""A batch's captured graph stays valid while its plans are used alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import synth  # noqa: E402
import paper_1107_2516_gb300 as dd  # noqa: E402


def beams(dtype, sigma=5.0):
    # few blocks: alone these plans launch more, smaller blocks than in the batch's grid
    plans, ins, outs = [], [], []
    for nch, step, ndm, nsamp in ((128, 0.1, 41, 8192), (256, 0.01, 64, 9000)):
        p = dd.Plan(nch, 150.0, -12.0 / nch, 327.68e-6, [step * i for i in range(ndm)], [1, 2, 4], sigma,
                    dd.DD_U8 if dtype == "u8" else dd.DD_F32, nsamp)
        x = synth.noise_f32(nch, nsamp, nch, pitch=9216)
        x[:, 4000:4003] += 2.0
        ins.append(torch.from_numpy(synth.quantize_u8(x) if dtype == "u8" else x).cuda())
        outs.append(torch.zeros(ndm * p.nsamp_out, dtype=torch.int32 if dtype == "u8" else torch.float32, device="cuda"))
        plans.append(p)
    return plans, ins, outs


def results(batch, plans, s, capacity=1 << 16):
    batch.launch(s)
    got = []
    for i, p in enumerate(plans):
        c, n = batch.results(i, capacity=capacity, stream=s)
        got.append((np.sort(c, order=("dm_idx", "t", "width_idx")), n, p.stats()))
    return got


def same(a, b):
    return all(np.array_equal(x[0], y[0]) and x[1:] == y[1:] for x, y in zip(a, b))


@pytest.mark.parametrize("dtype", ["f32", "u8"])
def test_replay_after_the_plans_ran_alone(dtype):
    # alone a plan needs more partial-statistics records than the graph was captured with
    plans, ins, outs = beams(dtype)
    s = torch.cuda.Stream()
    batch = dd.Batch(plans)
    batch.capture(ins, [9216] * 2, outs, s)
    first = results(batch, plans, s)
    assert all(n > 0 for _, n, _ in first)
    for p, x, o in zip(plans, ins, outs):
        p.execute(x, 9216, torch.empty_like(o))
        p.set_kernel(1)
        p.execute(x, 9216, torch.empty_like(o))
    torch.cuda.synchronize()
    fill = [torch.full((1 << k,), 255, dtype=torch.uint8, device="cuda") for k in range(10, 22)]   # takes what was freed
    second = results(batch, plans, s)
    assert same(first, second)
    assert all(bool((f == 255).all()) for f in fill)
    batch.close()
    for p in plans:
        p.close()


@pytest.mark.parametrize("dtype", ["f32", "u8"])
def test_replay_after_a_larger_search(dtype):
    # a search with room for more candidates than the graph was captured with
    plans, ins, outs = beams(dtype)
    s = torch.cuda.Stream()
    batch = dd.Batch(plans)
    batch.capture(ins, [9216] * 2, outs, s)
    first = results(batch, plans, s)
    other = []
    for p, x, o in zip(plans, ins, outs):
        out = torch.zeros_like(o)
        p.execute(x, 9216, out)
        out.zero_()                                # what the plan's own search finds last is not the batch's
        other.append(p.search(out, capacity=1 << 20)[1])
    torch.cuda.synchronize()
    fill = [torch.full((1 << k,), 255, dtype=torch.uint8, device="cuda") for k in range(10, 23)]
    second = results(batch, plans, s)
    assert same(first, second) and all(n != m for (_, n, _), m in zip(first, other))
    assert all(bool((f == 255).all()) for f in fill)
    # run directly, the batch takes the plans' buffers of now
    batch.execute(ins, [9216] * 2, outs)
    for i, p in enumerate(plans):
        c, n = batch.results(i)
        assert n == first[i][1] and np.array_equal(c, first[i][0])
    batch.close()
    for p in plans:
        p.close()
