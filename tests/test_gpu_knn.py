"""The seeding search (csrc/ff_seed_tc.cuh: tiles on the tensor cores, then the
eight best tiles' candidates) against the oracle: all integers, tolerance 0."""
from __future__ import annotations

import numpy as np
import pytest

import oracle as O
from paper_1703_02563_gb300 import ff

pytestmark = pytest.mark.gpu


def _frames(kind, C, W, H, seed):
    r = np.random.default_rng(seed)
    if kind == "noise":        # no structure
        return r.integers(0, 256, (2, C, H, W), dtype=np.uint8)
    if kind == "constant":     # every distance is 0: only the index ranks
        return np.full((2, C, H, W), 77, np.uint8)
    if kind == "stripes":      # few different vectors, many candidates each
        f = np.zeros((2, C, H, W), np.uint8)
        f[..., (np.arange(W) // 16) % 2 == 1] = 200
        f[1] = np.roll(f[1], 5, axis=-1)
        return f
    smooth = r.integers(0, 256, (2, C, H // 8 + 2, W // 8 + 2)).astype(np.float64)
    f = np.kron(smooth, np.ones((1, 1, 8, 8)))[:, :, :H, :W]
    f = f + r.integers(-6, 7, f.shape)
    return np.clip(f, 0, 255).astype(np.uint8)


CASES = [("smooth", 1, 1, 1, 1, 8, 1), ("smooth", 3, 31, 1, 1, 8, 1), ("smooth", 1, 33, 1, 2, 4, 1),
         ("smooth", 3, 32, 32, 2, 8, 1), ("smooth", 1, 41, 25, 2, 8, 1),
         # several chunks of tiles, ragged last tile; an odd stride
         ("smooth", 3, 430, 310, 4, 8, 1), ("smooth", 1, 257, 190, 3, 5, 3),
         # noise, where no two candidates are near:
         # one and several tiles of 128 queries, one chunk and many
         ("noise", 3, 256, 192, 3, 8, 1), ("noise", 1, 256, 192, 4, 8, 1),
         ("noise", 1, 300, 200, 2, 8, 1), ("noise", 3, 400, 300, 3, 8, 2),
         ("constant", 1, 200, 150, 3, 8, 1), ("stripes", 3, 160, 120, 3, 8, 1),
         ("stripes", 1, 200, 90, 2, 3, 1)]


@pytest.mark.parametrize("kind,C,W,H,S,leaf,stride", CASES)
@pytest.mark.parametrize("tc", [1, 0])
def test_seed_lists_equal_the_oracle(kind, C, W, H, S, leaf, stride, tc):
    import torch
    f = _frames(kind, C, W, H, W * 1000 + H)
    ctx = ff.Context(ff.Config(channels=C, scales=S, iters=1, seed_leaf=leaf, seed_stride=stride,
                               max_width=W + 3, max_height=H + 1))
    ff.ff_debug_set(ctx.ctx, ff.FF_DEBUG_SEED_TC, tc)
    for slot in (0, 1):
        ctx.features(slot, torch.from_numpy(f[slot]).cuda())
    f1, f2 = (O.features_all(f[k], S)[0] for k in (0, 1))
    for d, (a, b) in enumerate(((f1, f2), (f2, f1))):
        idx, dist = ctx.seed_knn(d)
        ridx, rdist = O.seed_knn(a, b, S, leaf, stride)
        np.testing.assert_array_equal(idx.cpu().numpy(), ridx)
        np.testing.assert_array_equal(dist.cpu().numpy(), rdist)
    # and a match seeded by it: the rerank at the coarsest scale
    flow, cost = ctx.match(0, 1, until_level=S - 1, until_sweeps=0)
    P = O.Params(channels=C, scales=S, iters=1, seed_leaf=leaf, seed_stride=stride)
    rf, rc, _ = O.match(P, f[0], f[1], 0, 1, until_level=S - 1, until_sweeps=0)
    np.testing.assert_array_equal(flow.cpu().numpy(), rf)
    np.testing.assert_array_equal(cost.cpu().numpy(), rc)
    ctx.sync()
    ctx.close()


def test_allocation_free_search_with_long_tiles():
    # as many queries as its scratch takes: two chunks, tiles of 512 candidates
    import torch
    W = H = 1448
    f = torch.from_numpy(_frames("smooth", 1, W, H, 4)).cuda()
    ctx = ff.Context(ff.Config(channels=1, scales=3, iters=1, max_width=W, max_height=H))
    feat = []
    for slot in (0, 1):
        ctx.features(slot, f[slot])
        x = torch.zeros((H, W, 16), dtype=torch.int8, device="cuda")
        x[..., :9] = ctx.features_of(slot, 0)
        feat.append(x)
    idx, dist = ctx.seed_knn(0)
    got_i, got_d = torch.empty_like(idx), torch.empty_like(dist)
    ff.ff_seed_knn_static(feat[0], feat[1], W, H, 1, 3, 8, 1, got_i, got_d,
                          torch.cuda.current_stream())
    assert torch.equal(got_i, idx) and torch.equal(got_d, dist)
    ctx.close()


@pytest.mark.parametrize("C,W,H,offset", [(3, 37, 29, 0), (3, 37, 29, 1), (1, 131, 3, 2), (1, 1, 1, 3)])
def test_feature_read_out_at_any_alignment(C, W, H, offset):
    import torch
    f = _frames("noise", C, W, H, 8)
    ctx = ff.Context(ff.Config(channels=C, scales=1, iters=1, max_width=W, max_height=H))
    ctx.features(0, torch.from_numpy(f[0]).cuda())
    buf = torch.full((W * H * 9 * C + 8,), 99, dtype=torch.int8, device="cuda")
    ff.ff_get_features(ctx.ctx, 0, 0, buf[offset:])
    got = buf.cpu().numpy()
    n = W * H * 9 * C
    np.testing.assert_array_equal(got[offset:offset + n],
                                  O.features_all(f[0], 1)[0].reshape(-1))
    assert (got[:offset] == 99).all() and (got[offset + n:] == 99).all()
    ctx.close()


@pytest.mark.parametrize("offset", [1, 2, 3])
def test_search_writes_arrays_at_any_alignment(offset):
    import torch
    W, H, leaf = 61, 43, 5
    f = torch.from_numpy(_frames("smooth", 3, W, H, 6)).cuda()
    ctx = ff.Context(ff.Config(channels=3, scales=2, iters=1, seed_leaf=leaf, max_width=W,
                               max_height=H))
    for slot in (0, 1):
        ctx.features(slot, f[slot])
    want = ctx.seed_knn(0)
    n = want[0].numel() * 4
    buf = torch.full((2, n + 16), 99, dtype=torch.uint8, device="cuda")
    ff.ff_seed_knn(ctx.ctx, 0, buf[0].data_ptr() + offset, buf[1].data_ptr() + 4 + offset)
    ctx.sync()
    for row, o, w in zip(buf.cpu().numpy(), (offset, 4 + offset), want):
        np.testing.assert_array_equal(row[o:o + n], w.cpu().numpy().reshape(-1).view(np.uint8))
        assert (row[:o] == 99).all() and (row[o + n:] == 99).all()
    ctx.close()


@pytest.mark.parametrize("C,S", [(1, 4), (3, 2)])
def test_search_with_the_shortest_wait_limit_ends_and_recovers(C, S):
    # whether a wait runs out is up to the load: each search either reports it or is right,
    # and the next one with the usual limit is right
    import torch
    W, H = 640, 200
    f = torch.from_numpy(_frames("smooth", C, W, H, 9)).cuda()
    ctx = ff.Context(ff.Config(channels=C, scales=S, iters=1, max_width=W, max_height=H))
    for slot in (0, 1):
        ctx.features(slot, f[slot])
    want = ctx.seed_knn(0)
    ctx.sync()
    for limit in (1000, 1000, 1000, 2_000_000_000):
        ff.ff_debug_set(ctx.ctx, ff.FF_DEBUG_WAIT_LIMIT_NS, limit)
        got = ctx.seed_knn(0)
        try:
            ctx.sync()
        except ff.FFError as e:
            assert e.status == ff.FF_ETIMEOUT and limit == 1000
            continue
        for a, b in zip(got, want):
            assert torch.equal(a, b)
    ctx.close()


# tiles of 32 candidates up to 256 x 128 of them, of 128 above: both sides of the line, several
# chunks, ragged last tiles; and every case above through the allocation-free search
FINE = [("smooth", 1, 256, 128, 3, 8, 1), ("smooth", 1, 331, 99, 3, 8, 1), ("smooth", 3, 257, 128, 3, 8, 1),
        ("noise", 3, 331, 198, 4, 8, 2), ("noise", 1, 9, 7, 1, 8, 2), ("stripes", 3, 640, 480, 4, 8, 8)]


@pytest.mark.parametrize("kind,C,W,H,S,leaf,stride", FINE)
def test_lists_at_the_line_between_tile_sizes(kind, C, W, H, S, leaf, stride):
    test_seed_lists_equal_the_oracle(kind, C, W, H, S, leaf, stride, 1)


# equal candidates, where the ranking ends at the first tile that cannot hold a better one: tiles
# of 32 and of 128, strides, two halves of one vector each
TIES = [("constant", 3, 331, 99, 2, 8, 4), ("constant", 1, 331, 199, 3, 5, 1), ("stripes", 1, 331, 99, 2, 8, 3),
        ("stripes", 3, 333, 201, 4, 7, 1)]


@pytest.mark.parametrize("kind,C,W,H,S,leaf,stride", TIES)
def test_lists_of_equal_candidates(kind, C, W, H, S, leaf, stride):
    test_seed_lists_equal_the_oracle(kind, C, W, H, S, leaf, stride, 1)


@pytest.mark.parametrize("kind,C,W,H,S,leaf,stride", CASES + FINE + TIES)
def test_allocation_free_search_equals_the_oracle(kind, C, W, H, S, leaf, stride):
    import torch
    f = _frames(kind, C, W, H, W * 1000 + H)
    f1, f2 = (O.features_all(f[k], S)[0] for k in (0, 1))
    P = 16 if C == 1 else 32
    feat = []
    for x in (f1, f2):
        y = torch.zeros((H, W, P), dtype=torch.int8, device="cuda")
        y[..., :9 * C] = torch.from_numpy(np.ascontiguousarray(x).reshape(H, W, 9 * C)).cuda()
        feat.append(y)
    ridx, rdist = O.seed_knn(f1, f2, S, leaf, stride)
    idx = torch.empty(ridx.shape, dtype=torch.int32, device="cuda")
    dist = torch.empty_like(idx)
    ff.ff_seed_knn_static(feat[0], feat[1], W, H, C, S, leaf, stride, idx, dist,
                          torch.cuda.current_stream())
    np.testing.assert_array_equal(idx.cpu().numpy(), ridx)
    np.testing.assert_array_equal(dist.cpu().numpy(), rdist)
