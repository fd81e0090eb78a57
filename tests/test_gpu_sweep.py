"""The sweep kernel (E2M1 triangles of ibs_compute) at its own edges, against the
oracle: half-blocks of 64 samples, row pairs of 256, column groups of 384, ring
stages of 288 markers, rows at every alignment, tiles split into parts and
whole waves of tiles; the call whose workspace has no room for it; and the gather
of batched subsets from both forms of the pool."""
import numpy as np
import pytest

import oracle
from helpers import assert_dist_close, gpu_compute, pack_codes, random_codes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1410_4803_gb300 import ibs
    c = ibs.ibs_init(0, flags=ibs.IBS_KERNEL_TC | ibs.IBS_TC_FP4)
    yield c
    ibs.ibs_shutdown(c)


def _check(ctx, n, m, seed):
    rng = np.random.default_rng(seed)
    packed = pack_codes(random_codes(rng, n, m, miss=0.05), garbage_rng=rng)
    want_c, want_d = oracle.ibs_triangle(packed, n, m)
    got_c, got_d = gpu_compute(ctx, packed, n, m)
    bad = np.flatnonzero((got_c != want_c).any(axis=1))
    assert bad.size == 0, f"n={n} m={m}: {bad.size} pairs differ, first {bad[:5]}"
    assert_dist_close(got_d, want_d)


@pytest.mark.parametrize("n", [1, 64, 65, 192, 193, 255, 257, 384, 385, 511, 513, 639, 770])
@pytest.mark.parametrize("m", [1, 31, 287, 288, 289, 577, 2593])
def test_edges(ctx, n, m):
    _check(ctx, n, m, 1000 * n + m)


# parts only (few tiles, many markers; many tiles, few markers); one full wave of whole tiles (76 clusters) and
# a split rest; two waves, with more than one lockstep segment each
@pytest.mark.parametrize("n,m", [(130, 60_000), (1100, 9_001), (3201, 2_000), (4500, 3_003), (3000, 1_000), (3000, 50)])
def test_parts_and_waves(ctx, n, m):
    _check(ctx, n, m, n + m)


# either side of the sizes that leave the sweep kernel: one block of samples, two
# (the two-SM kernel from 65,536 markers on)
@pytest.mark.parametrize("n,m", [(128, 16_384), (128, 16_385), (129, 16_385), (256, 49_152), (256, 49_153), (257, 49_153),
                                 (200, 70_000), (72, 10_368), (72, 10_369), (129, 32_135), (129, 32_136), (20, 1299)])
def test_narrow_inputs(ctx, n, m):
    _check(ctx, n, m, n + m)


# either side of the markers that a call without distances needs for the sweep kernel
@pytest.mark.parametrize("n,m", [(128, 1300), (500, 2000), (2048, 3500), (2300, 65)])
@pytest.mark.parametrize("square", [False, True])
def test_counts_alone(n, m, square):
    import torch
    from paper_1410_4803_gb300 import ibs
    c = ibs.ibs_init(0, flags=ibs.IBS_KERNEL_TC | ibs.IBS_TC_FP4 | (ibs.IBS_OUT_SQUARE if square else 0))
    try:
        for mm in (m - 1, m) if not square else (1299, 1300):
            rng = np.random.default_rng(n + mm)
            packed = pack_codes(random_codes(rng, n, mm, miss=0.05))
            want = oracle.ibs_triangle(packed, n, mm)[0]
            counts = torch.full((n * n if square else n * (n + 1) // 2, 4), -7, dtype=torch.int32, device="cuda")
            ibs.ibs_compute(c, torch.from_numpy(packed).cuda(), n, mm, counts)
            ibs.ibs_synchronize(c)
            got = counts.cpu().numpy()
            if square:
                i, j = np.triu_indices(n)
                got = got.reshape(n, n, 4)
                assert (got[j, i] == want).all()
                got = got[i, j]
            assert (got == want).all(), mm
    finally:
        ibs.ibs_shutdown(c)


# planes 26 MB, partial counts 2.9 MB: the one-SM kernel; planes 51 MB: the two-SM kernel
@pytest.mark.parametrize("n,m,limit,kernel", [(600, 20_000, 32 << 20, "tc-persistent"), (300, 66_000, 56 << 20, "tc-pair")])
def test_no_room_for_the_workspace(n, m, limit, kernel):
    """A workspace bound that holds operand planes and partial counts but not
    the sweep kernel's scratch and parts: the call still computes."""
    from paper_1410_4803_gb300 import ibs
    rng = np.random.default_rng(3)
    packed = pack_codes(random_codes(rng, n, m))
    want_c, want_d = oracle.ibs_triangle(packed, n, m)
    c = ibs.ibs_init(0, workspace_bytes=limit)
    try:
        assert ibs.ibs_compute_kernel(c, n, m) == kernel and ibs.ibs_compute_sweep_kernel(c, n, m)
        for _ in range(2):
            got_c, got_d = gpu_compute(c, packed, n, m)
            assert not ibs.ibs_compute_sweep_kernel(c, n, m)
            assert (got_c == want_c).all()
            assert_dist_close(got_d, want_d)
    finally:
        ibs.ibs_shutdown(c)


def test_shapes_without_room_are_remembered():
    """Calls of two such shapes in turn try the sweep kernel's workspace once
    each, not on every call (a device-wide free and allocation each time)."""
    from paper_1410_4803_gb300 import ibs
    rng = np.random.default_rng(4)
    shapes = [(600, 20_000), (500, 20_000)]
    packed = [pack_codes(random_codes(rng, n, m)) for n, m in shapes]
    want = [oracle.ibs_triangle(p, n, m)[0] for p, (n, m) in zip(packed, shapes)]
    c = ibs.ibs_init(0, workspace_bytes=32 << 20)
    try:
        for _ in range(2):
            for p, (n, m), w in zip(packed, shapes, want):
                assert (gpu_compute(c, p, n, m)[0] == w).all()
        assert not any(ibs.ibs_compute_sweep_kernel(c, n, m) for n, m in shapes)
    finally:
        ibs.ibs_shutdown(c)


@pytest.mark.parametrize("pool_n,n,vb,vl", [
    (1003, 1000, 0, 3001),   # the window regrouped by sample: from the first marker to the last
    (1003, 300, 37, 2593),   # from inside a column of the pool
    (1003, 251, 2968, 33),   # two columns, just above a quarter of the pool's samples
    (1003, 250, 37, 2593),   # below a quarter: single bytes
    (4096, 1, 0, 3001),
])
def test_batch_gather(ctx, pool_n, n, vb, vl):
    import torch
    from paper_1410_4803_gb300 import ibs
    rng = np.random.default_rng(n + vl)
    codes = random_codes(rng, pool_n, 3001, miss=0.05)
    idx = rng.permutation(pool_n)[:n].astype(np.int64)
    want_c, want_d = oracle.ibs_triangle(pack_codes(codes[idx][:, vb:vb + vl]), n, vl)
    pool = torch.from_numpy(pack_codes(codes, garbage_rng=rng)).cuda()
    dev_idx = torch.from_numpy(idx).cuda()
    for _ in range(2):
        out_c = torch.full((n * (n + 1) // 2, 4), -7, dtype=torch.int32, device="cuda")
        out_d = torch.empty(n * (n + 1) // 2, dtype=torch.float64, device="cuda")
        ibs.ibs_compute_batch(ctx, pool, pool_n, 3001, [(dev_idx, vb, vl, out_c, out_d)])
        ibs.ibs_synchronize(ctx)
        assert (out_c.cpu().numpy() == want_c).all()
        assert_dist_close(out_d.cpu().numpy(), want_d)


# the mirror image at the edges of row pairs, column groups and pieces; parts and
# whole tiles.  The distances are the IEEE quotients.
@pytest.mark.parametrize("n,m", [(1, 31), (129, 289), (257, 1000), (385, 2593), (513, 577), (1100, 9_001), (3201, 600)])
def test_square(ctx, n, m):
    from paper_1410_4803_gb300 import ibs
    rng = np.random.default_rng(n + m)
    packed = pack_codes(random_codes(rng, n, m, miss=0.05))
    tri_c, tri_d = gpu_compute(ctx, packed, n, m)
    sq = ibs.ibs_init(0, flags=ibs.IBS_KERNEL_TC | ibs.IBS_TC_FP4 | ibs.IBS_OUT_SQUARE)
    try:
        got_c, got_d = gpu_compute(sq, packed, n, m, square=True)
    finally:
        ibs.ibs_shutdown(sq)
    got_c, got_d = got_c.reshape(n, n, 4), got_d.reshape(n, n)
    i, j = np.triu_indices(n)
    for c, d in ((got_c[i, j], got_d[i, j]), (got_c[j, i], got_d[j, i])):
        assert (c == tri_c).all()
        np.testing.assert_array_equal(d, tri_d)
    c = tri_c.astype(np.float64)
    with np.errstate(invalid="ignore"):
        np.testing.assert_array_equal(tri_d, (c[:, 1] + 2 * c[:, 0]) / (2 * c[:, 3]))


@pytest.mark.parametrize("n,m", [(130, 1_000), (3201, 600)])  # parts only; whole waves with lockstep counters
def test_recorded_into_a_graph(ctx, n, m):
    """A call of a shape seen before, captured and replayed on new genotypes."""
    import torch
    from paper_1410_4803_gb300 import ibs
    rng = np.random.default_rng(n)
    packed = torch.from_numpy(pack_codes(random_codes(rng, n, m))).cuda()
    counts = torch.empty((n * (n + 1) // 2, 4), dtype=torch.int32, device="cuda")
    dist = torch.empty(n * (n + 1) // 2, dtype=torch.float64, device="cuda")
    ibs.ibs_compute(ctx, packed, n, m, counts, dist)
    ibs.ibs_synchronize(ctx)
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        ibs.ibs_compute(ctx, packed, n, m, counts, dist, stream=stream)
    again = pack_codes(random_codes(rng, n, m, miss=0.1))
    packed.copy_(torch.from_numpy(again))
    counts.fill_(-7)
    graph.replay()
    torch.cuda.synchronize()
    want_c, want_d = oracle.ibs_triangle(again, n, m)
    assert (counts.cpu().numpy() == want_c).all()
    assert_dist_close(dist.cpu().numpy(), want_d)
