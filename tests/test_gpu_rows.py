"""Serving steps of few rows (code bits of the panel, population counts) and the
top-k selection, at their own edges, against the oracle: row groups of 1, 2, 4
and 8, 512 panel samples per CTA, staged pieces of 64 columns of 32 markers;
rows whose nearest samples tie past the selection's candidate list."""
import numpy as np
import pytest

import oracle
from helpers import pack_codes, random_codes

pytestmark = pytest.mark.gpu


def _query(ctx, packed, q, n, k):
    import torch
    from paper_1410_4803_gb300 import ibs
    counts = torch.full((q, n, 4), -7, dtype=torch.int32, device="cuda")
    idx = torch.empty((q, k), dtype=torch.int32).pin_memory()
    dist = torch.empty((q, k), dtype=torch.float64).pin_memory()
    ibs.ibs_wait(ctx, ibs.ibs_query(ctx, torch.from_numpy(packed).pin_memory(), q, k, counts, idx, dist))
    return counts.cpu().numpy(), idx.numpy(), dist.numpy()


def _expected(panel, rows):
    """Counts [q][n][4] of rows against the panel, by the oracle's triangle of both."""
    n, q = panel.shape[0], rows.shape[0]
    counts, _ = oracle.ibs_triangle(pack_codes(np.concatenate([rows, panel])), n + q, panel.shape[1])
    at = lambda i: i * (n + q) - i * (i - 1) // 2 + np.arange(q, q + n) - i  # noqa: E731
    return np.stack([counts[at(i)] for i in range(q)])


def _check_topk(counts, idx, dist, k):
    for c, got_i, got_d in zip(counts.astype(np.float64), idx, dist):
        with np.errstate(invalid="ignore"):
            d = (c[:, 1] + 2 * c[:, 0]) / (2 * c[:, 3])
        order = np.lexsort((np.arange(d.size), np.where(np.isnan(d), np.inf, d)))[:k]
        assert (got_i[:order.size] == order).all()
        np.testing.assert_array_equal(got_d[:order.size], d[order])  # NaN equal
        assert (got_i[order.size:] == -1).all() and np.isnan(got_d[order.size:]).all()


def _run(panel, rows, k):
    from paper_1410_4803_gb300 import ibs
    ctx = ibs.ibs_init(0, flags=ibs.IBS_KERNEL_TC | ibs.IBS_TC_FP4)
    try:
        ibs.ibs_panel_load(ctx, pack_codes(panel), panel.shape[0], panel.shape[1])
        for _ in range(2):
            got, idx, dist = _query(ctx, pack_codes(rows), rows.shape[0], panel.shape[0], k)
            want = _expected(panel, rows)
            assert (got == want).all()
            _check_topk(want, idx, dist, k)
    finally:
        ibs.ibs_shutdown(ctx)


@pytest.mark.parametrize("q", [1, 2, 3, 4, 5, 8, 9, 16, 17])
@pytest.mark.parametrize("n,m", [(1, 31), (255, 2049), (512, 2048), (513, 33), (1025, 4097)])
def test_few_rows(q, n, m):
    rng = np.random.default_rng(q * 10007 + n + m)
    _run(random_codes(rng, n, m, miss=0.05), random_codes(rng, q, m, miss=0.05), min(16, 2 * n))


# 8 rows on the code bits, 9 on the operand planes of a panel past the size for more
@pytest.mark.parametrize("q", [8, 9])
def test_few_rows_of_a_larger_panel(q):
    import torch
    from paper_1410_4803_gb300 import ibs
    rng = np.random.default_rng(q)
    n, m = 2003, 200_003
    packed = rng.integers(0, 256, (m, (n + 3) // 4), dtype=np.uint8)
    rows = rng.integers(0, 256, (m, (q + 3) // 4), dtype=np.uint8)
    ctx = ibs.ibs_init(0, flags=ibs.IBS_KERNEL_TC | ibs.IBS_TC_FP4)
    try:
        ibs.ibs_panel_load(ctx, torch.from_numpy(packed).cuda(), n, m)
        got, idx, dist = _query(ctx, rows, q, n, 16)
    finally:
        ibs.ibs_shutdown(ctx)
    want = oracle.ibs_block(oracle.unpack(rows, q, m), oracle.unpack(packed, n, m))[0]
    assert (got == want).all()
    _check_topk(want, idx, dist, 16)


# two markers: few distinct distances, and rows without a common call
@pytest.mark.parametrize("q", [1, 40])
@pytest.mark.parametrize("n,k", [(3, 64), (127, 64), (600, 1), (3000, 64), (3000, 16)])
def test_topk_ties(q, n, k):
    rng = np.random.default_rng(q + n + k)
    _run(random_codes(rng, n, 2, miss=0.3), random_codes(rng, q, 2, miss=0.3), k)


@pytest.mark.parametrize("skew", [1, 4])
def test_topk_lists_at_any_alignment(skew):
    """Pinned lists that a kernel could not store to element by element are still copied there."""
    import torch
    from paper_1410_4803_gb300 import ibs
    rng = np.random.default_rng(skew)
    n, m, q, k = 300, 700, 3, 8
    panel, rows = random_codes(rng, n, m), random_codes(rng, q, m)
    ctx = ibs.ibs_init(0, flags=ibs.IBS_KERNEL_TC | ibs.IBS_TC_FP4)
    try:
        ibs.ibs_panel_load(ctx, pack_codes(panel), n, m)
        idx = torch.zeros(q * k * 4 + 16, dtype=torch.uint8).pin_memory()
        dist = torch.zeros(q * k * 8 + 16, dtype=torch.uint8).pin_memory()
        packed = torch.from_numpy(pack_codes(rows)).pin_memory()
        ibs.ibs_wait(ctx, ibs.ibs_query(ctx, packed, q, k, None, idx.data_ptr() + skew, dist.data_ptr() + skew))
        got_i = np.frombuffer(idx.numpy().tobytes()[skew:skew + q * k * 4], np.int32).reshape(q, k)
        got_d = np.frombuffer(dist.numpy().tobytes()[skew:skew + q * k * 8], np.float64).reshape(q, k)
        _check_topk(_expected(panel, rows), got_i, got_d, k)
    finally:
        ibs.ibs_shutdown(ctx)
