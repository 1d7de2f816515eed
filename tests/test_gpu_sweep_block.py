"""The sweep by blocks of four columns (csrc/ff_block.cuh) at the edges of its blocks,
strips and clusters, under graph capture, and against the batch sweep: all integers,
tolerance 0."""
from __future__ import annotations

import numpy as np
import pytest

import oracle as O
from paper_1703_02563_gb300 import ff, workloads

pytestmark = pytest.mark.gpu


def _run(ctx, pair, pair_id, **kw):
    import torch
    for slot, img in ((0, pair.img1), (1, pair.img2)):
        ctx.features(slot, torch.from_numpy(np.ascontiguousarray(img)).cuda())
    return [[t.cpu().numpy() for t in ctx.match(d, pair_id, **kw)] for d in (0, 1)]


# columns: below, at and past a block, the 16-block ring, the 512 columns up to which
# launches overlap; rows: below, at and past a strip (4) and a cluster (32), and the
# second cluster's loader at ragged widths
@pytest.mark.parametrize("C,W,H", [(1, 3, 5), (3, 4, 4), (1, 5, 33), (3, 6, 32), (3, 7, 66),
                                   (1, 64, 31), (3, 65, 33), (1, 67, 37), (3, 130, 35),
                                   (1, 515, 9), (3, 514, 34)])
def test_every_sweep_equals_the_oracle(C, W, H):
    pair = workloads.random_pair(seed=W * 100 + H, width=W, height=H, channels=C)
    S, I = 2, 5     # all four directions and the first again
    ctx = ff.Context(ff.Config(channels=C, scales=S, iters=I, radius_q3=12, max_width=W + 2,
                               max_height=H))
    P = O.Params(channels=C, scales=S, iters=I, radius_q3=12)
    for L in (1, 0):
        for k in range(I + 1):
            got = _run(ctx, pair, 7, until_level=L, until_sweeps=k)
            for d, (a, b) in enumerate(((pair.img1, pair.img2), (pair.img2, pair.img1))):
                rf, rc, _ = O.match(P, a, b, d, 7, until_level=L, until_sweeps=k)
                np.testing.assert_array_equal(got[d][0], rf, err_msg=f"dir {d} L {L} k {k}")
                np.testing.assert_array_equal(got[d][1], rc, err_msg=f"dir {d} L {L} k {k}")
    ctx.sync()
    ctx.close()


@pytest.mark.parametrize("C", [1, 3])
def test_captured_match_replays(C):
    import torch
    pair = workloads.random_pair(seed=C, width=150, height=70, channels=C)
    ctx = ff.Context(ff.Config(channels=C, scales=3, iters=4, max_width=150, max_height=70))
    want = _run(ctx, pair, 3)[0]
    flow = torch.empty((70, 150, 2), dtype=torch.int16, device="cuda")
    cost = torch.empty((70, 150), dtype=torch.int32, device="cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    ff.ff_set_stream(ctx.ctx, s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        ff.ff_match(ctx.ctx, 0, 3, None, flow, cost)
    for _ in range(3):
        flow.fill_(1)
        cost.fill_(1)
        g.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(flow.cpu().numpy(), want[0])
        np.testing.assert_array_equal(cost.cpu().numpy(), want[1])
    ff.ff_set_stream(ctx.ctx, torch.cuda.current_stream())
    ctx.close()


@pytest.mark.parametrize("schedule", [ff.FF_SCHED_PLUS, ff.FF_SCHED_PLUS_FAST_X2])
def test_block_and_batch_sweeps_agree_on_large_frames(schedule):
    pair = workloads.random_pair(seed=5, width=1301, height=401, channels=3)
    ctx = ff.Context(ff.Config(channels=3, scales=4, radius_q3=8, seed_stride=3, schedule=schedule,
                               max_width=1301, max_height=401))
    got = {}
    for lanes in (4, 2):
        ff.ff_debug_set(ctx.ctx, ff.FF_DEBUG_SWEEP_LANES, lanes)
        got[lanes] = _run(ctx, pair, 1)
    for d in (0, 1):
        for a, b in zip(got[4][d], got[2][d]):
            np.testing.assert_array_equal(a, b)
    ctx.sync()
    ctx.close()


# one expired wait ends the match: its other CTAs (of the tall frame not all fit the GPU at
# once) and its later sweeps do not wait for their own limit
@pytest.mark.parametrize("C,W,H,S", [(1, 128, 96, 3), (3, 128, 96, 3), (1, 64, 4096, 1)])
def test_an_expired_wait_ends_the_match(C, W, H, S):
    import time

    import torch
    limit = 0.25
    pair = workloads.random_pair(seed=C, width=W, height=H, channels=C)
    ctx = ff.Context(ff.Config(channels=C, scales=S, iters=4, seed_stride=8, max_width=W,
                               max_height=H))
    want = _run(ctx, pair, 1)
    ctx.sync()
    ff.ff_debug_set(ctx.ctx, ff.FF_DEBUG_WAIT_LIMIT_NS, int(limit * 1e9))
    ff.ff_debug_set(ctx.ctx, ff.FF_DEBUG_FORCE_TIMEOUT, 1)
    torch.cuda.synchronize()
    start = time.perf_counter()
    ctx.match(0, 1)
    with pytest.raises(ff.FFError) as e:
        ctx.sync()
    took = time.perf_counter() - start
    assert e.value.status == ff.FF_ETIMEOUT
    assert limit <= took < 2 * limit
    ff.ff_debug_set(ctx.ctx, ff.FF_DEBUG_FORCE_TIMEOUT, 0)
    for a, b in zip(_run(ctx, pair, 1), want):
        for x, y in zip(a, b):
            np.testing.assert_array_equal(x, y)
    ctx.sync()
    ctx.close()
