"""Batched path (ibs_compute_batch): many subsets of a pool over uneven
variant windows in one persistent launch under a CUDA graph.  Each subset's
result must equal the plain path on that subset alone and the oracle."""
import numpy as np
import pytest

import oracle
from helpers import assert_dist_close, pack_codes

pytestmark = pytest.mark.gpu


def _subset_packed(pool_codes, idx, vb, vl):
    return pack_codes(pool_codes[idx][:, vb:vb + vl])


@pytest.fixture(scope="module")
def pool():
    from paper_1410_4803_gb300 import synth
    w = synth.batch_pool(pool_n=1500, pool_m=30000, seed=11)
    codes = oracle.unpack(w.packed, w.n, w.m)
    return w, codes


def _make_subsets(rng, pool_n, pool_m):
    spec = [(1, 1), (2, 31), (63, 33), (64, 385), (65, 1000), (130, 4097), (700, 20000), (257, 383),
            (5, 29999), (400, 12345), (129, 64), (900, 7000)]
    subs = []
    for n, vl in spec:
        idx = rng.choice(pool_n, size=n, replace=False).astype(np.int64)
        if rng.random() < 0.5:
            idx = np.sort(idx)
        vb = int(rng.integers(0, pool_m - vl + 1))
        subs.append((idx, vb, vl))
    return subs


def _run_batch(ctx, w, subs, dev_packed):
    import torch
    from paper_1410_4803_gb300 import ibs
    args, outs = [], []
    for idx, vb, vl in subs:
        n = idx.size
        P = n * (n + 1) // 2
        c = torch.full((P, 4), -7, dtype=torch.int32, device="cuda")
        d = torch.empty(P, dtype=torch.float64, device="cuda")
        it = torch.from_numpy(idx).cuda()
        args.append((it, vb, vl, c, d))
        outs.append((c, d, it))
    ibs.ibs_compute_batch(ctx, dev_packed, w.n, w.m, args)
    ibs.ibs_synchronize(ctx)
    return [(c.cpu().numpy(), d.cpu().numpy()) for c, d, _ in outs]


def test_batch_matches_plain_and_oracle(pool, tmp_path):
    import torch
    from paper_1410_4803_gb300 import ibs
    w, codes = pool
    rng = np.random.default_rng(5)
    subs = _make_subsets(rng, w.n, w.m)
    dev_packed = torch.from_numpy(w.packed).cuda()
    ctx = ibs.ibs_init(0, autotune_cache_path=str(tmp_path / "tune.jsonl"))
    plain = ibs.ibs_init(0)
    try:
        first = _run_batch(ctx, w, subs, dev_packed)
        second = _run_batch(ctx, w, subs, dev_packed)  # graph replay with new output buffers
        for (idx, vb, vl), (c1, d1), (c2, d2) in zip(subs, first, second):
            n = idx.size
            assert (c1 == c2).all()
            sp = _subset_packed(codes, idx, vb, vl)
            pc, pd = ibs.compute(plain, torch.from_numpy(sp).cuda(), n, vl)
            ibs.ibs_synchronize(plain)
            assert (c1 == pc.cpu().numpy()).all(), f"batch != plain for n={n} window={vb}+{vl}"
            G = oracle.unpack_subset(w.packed, w.n, w.m, idx, vb, vl)
            oc, od, _ = oracle.ibs_triangle_from_codes(G)
            assert (c1 == oc).all(), f"batch != oracle for n={n} window={vb}+{vl}"
            assert_dist_close(d1, od)
        info = ibs.ibs_batch_plan_info(ctx)
        assert info["items"] > 0 and info["grid"] > 0
        assert info["mode"] in (3, 4)  # tensor-core form by default, as ibs_compute
        assert (tmp_path / "tune.jsonl").exists()
    finally:
        ibs.ibs_shutdown(plain)
        ibs.ibs_shutdown(ctx)


def _flags(ibs, names):
    f = 0
    for nm in names.split("|"):
        f |= getattr(ibs, nm)
    return f


@pytest.mark.parametrize("flags_name", ["IBS_KERNEL_PLAIN", "IBS_KERNEL_CSA", "IBS_KERNEL_TC|IBS_TC_FP8",
                                        "IBS_KERNEL_TC|IBS_TC_FP4"])
def test_batch_forced_modes(pool, flags_name):
    import torch
    from paper_1410_4803_gb300 import ibs
    w, codes = pool
    rng = np.random.default_rng(6)
    subs = _make_subsets(rng, w.n, w.m)[:6]
    ctx = ibs.ibs_init(0, flags=_flags(ibs, flags_name))
    try:
        res = _run_batch(ctx, w, subs, torch.from_numpy(w.packed).cuda())
        for (idx, vb, vl), (c, d) in zip(subs, res):
            G = oracle.unpack_subset(w.packed, w.n, w.m, idx, vb, vl)
            oc, od, _ = oracle.ibs_triangle_from_codes(G)
            assert (c == oc).all()
    finally:
        ibs.ibs_shutdown(ctx)


@pytest.mark.parametrize("flags_name", ["IBS_KERNEL_CSA", "IBS_KERNEL_TC|IBS_TC_FP8", "IBS_KERNEL_TC|IBS_TC_FP4"])
def test_batch_split_items(pool, flags_name):
    """One subset of few tiles and many chunks: the autotuner splits the
    marker axis into items that add into a partial triangle, and a finalize
    launch writes the counts."""
    import torch
    from paper_1410_4803_gb300 import ibs
    w, _ = pool
    rng = np.random.default_rng(8)
    subs = [(np.sort(rng.choice(w.n, size=150, replace=False)).astype(np.int64), 17, 29000)]
    ctx = ibs.ibs_init(0, flags=_flags(ibs, flags_name))
    try:
        (c, d), = _run_batch(ctx, w, subs, torch.from_numpy(w.packed).cuda())
        # tensor-core modes may also pick the per-subset launches (policy 2),
        # which split this subset's few tiles over K as ibs_compute does
        assert ibs.ibs_batch_plan_info(ctx)["split_policy"] in ((1, 2, 3) if "TC" in flags_name else (1,))
        idx, vb, vl = subs[0]
        G = oracle.unpack_subset(w.packed, w.n, w.m, idx, vb, vl)
        oc, od, _ = oracle.ibs_triangle_from_codes(G)
        assert (c == oc).all()
        assert_dist_close(d, od)
    finally:
        ibs.ibs_shutdown(ctx)


@pytest.mark.parametrize("policy", [0, 1, 2, 3, 4, 5])
@pytest.mark.parametrize("fmt", ["IBS_TC_FP8", "IBS_TC_FP4"])
def test_batch_each_policy(pool, policy, fmt, monkeypatch):
    """Every split policy of the tensor-core batch, fixed by IBS_BATCH_POLICY:
    0 whole tiles in one launch per stage, 1 K-split large subsets, 2 one
    launch per subset over its own work list (small subsets and tail waves
    split over K, split tiles finalised from the subset descriptors), 3 and 4
    (E2M1 only) one launch of the two-SM kernel over every subset's pair items
    with the gather fused in, 5 (E2M1 only) policy 2's launches with each
    two-SM launch's epilogue warps gathering the following subsets (here every
    window is under the two-SM size, so each subset gets its own gather
    launch; the fused form is tested in a child below).  Counts equal the
    oracle for all twelve subsets, twice (graph replay)."""
    import torch
    from paper_1410_4803_gb300 import ibs
    if policy >= 3 and fmt != "IBS_TC_FP4":
        pytest.skip("the two-SM kernel takes E2M1 operands only")
    monkeypatch.setenv("IBS_BATCH_POLICY", str(policy))
    w, codes = pool
    rng = np.random.default_rng(9)
    subs = _make_subsets(rng, w.n, w.m)
    ctx = ibs.ibs_init(0, flags=_flags(ibs, "IBS_KERNEL_TC|" + fmt))
    try:
        dev = torch.from_numpy(w.packed).cuda()
        first = _run_batch(ctx, w, subs, dev)
        second = _run_batch(ctx, w, subs, dev)
        assert ibs.ibs_batch_plan_info(ctx)["split_policy"] == policy
        for (idx, vb, vl), (c1, d1), (c2, d2) in zip(subs, first, second):
            G = oracle.unpack_subset(w.packed, w.n, w.m, idx, vb, vl)
            oc, od, _ = oracle.ibs_triangle_from_codes(G)
            assert (c1 == oc).all(), f"policy {policy}: n={idx.size} window={vb}+{vl}"
            assert (c2 == oc).all()
            assert_dist_close(d1, od)
            np.testing.assert_array_equal(d1, d2)
    finally:
        ibs.ibs_shutdown(ctx)


def test_batch_policy2_without_the_sweep_kernel(pool, monkeypatch):
    """Policy 2's launches per subset, which the sweep kernel stands in for where it can run."""
    import torch
    from paper_1410_4803_gb300 import ibs
    monkeypatch.setenv("IBS_BATCH_POLICY", "2")
    monkeypatch.setenv("IBS_SWEEP", "0")
    w, codes = pool
    subs = _make_subsets(np.random.default_rng(9), w.n, w.m)
    ctx = ibs.ibs_init(0, flags=_flags(ibs, "IBS_KERNEL_TC|IBS_TC_FP4"))
    try:
        dev = torch.from_numpy(w.packed).cuda()
        for _ in range(2):
            res = _run_batch(ctx, w, subs, dev)
            assert ibs.ibs_last_launch_info(ctx)["launches"] > len(subs)
            for (idx, vb, vl), (c, d) in zip(subs, res):
                G = oracle.unpack_subset(w.packed, w.n, w.m, idx, vb, vl)
                oc, od, _ = oracle.ibs_triangle_from_codes(G)
                assert (c == oc).all(), f"n={idx.size} window={vb}+{vl}"
                assert_dist_close(d, od)
    finally:
        ibs.ibs_shutdown(ctx)


def test_batch_out_of_range_index_is_reported(pool):
    """A corrupted sample index is not read: the kernel treats that sample as
    all-missing and ibs_synchronize reports IBS_EINVAL."""
    import torch
    from paper_1410_4803_gb300 import ibs
    w, _ = pool
    ctx = ibs.ibs_init(0)
    try:
        idx = torch.tensor([0, 5, w.n + 100], dtype=torch.int64, device="cuda")
        c = torch.empty((6, 4), dtype=torch.int32, device="cuda")
        ibs.ibs_compute_batch(ctx, torch.from_numpy(w.packed).cuda(), w.n, w.m, [(idx, 0, 500, c, None)])
        with pytest.raises(ibs.IbsError) as ei:
            ibs.ibs_synchronize(ctx)
        assert ei.value.status == ibs.IBS_EINVAL
        got = c.cpu().numpy()
        # pairs with the bad sample have N = 0
        assert got[oracle.tri_index(0, 2, 3), 3] == 0 and got[oracle.tri_index(2, 2, 3), 3] == 0
    finally:
        ibs.ibs_shutdown(ctx)


def test_batch_validation_errors(pool):
    import torch
    from paper_1410_4803_gb300 import ibs
    w, _ = pool
    ctx = ibs.ibs_init(0)
    try:
        idx = torch.arange(10, dtype=torch.int64, device="cuda")
        c = torch.empty((55, 4), dtype=torch.int32, device="cuda")
        with pytest.raises(ibs.IbsError) as ei:
            ibs.ibs_compute_batch(ctx, torch.from_numpy(w.packed).cuda(), w.n, w.m, [(idx, w.m - 10, 20, c, None)])
        assert ei.value.status == ibs.IBS_EINVAL
    finally:
        ibs.ibs_shutdown(ctx)


def test_batch_windows_move_between_calls(pool):
    """Same subset shapes (n, window length) on two calls, but the windows
    start elsewhere on the second: the cached plan is reused and the gather's
    CTA map (ordered by pool variant) is rebuilt; both calls equal the oracle."""
    import torch
    from paper_1410_4803_gb300 import ibs
    w, _ = pool
    rng = np.random.default_rng(12)
    subs = _make_subsets(rng, w.n, w.m)[:8]
    moved = []
    for idx, vb, vl in subs:
        vb2 = int(rng.integers(0, w.m - vl + 1))
        moved.append((idx, vb2, vl))
    ctx = ibs.ibs_init(0)
    try:
        dev = torch.from_numpy(w.packed).cuda()
        for case in (subs, moved, subs):
            res = _run_batch(ctx, w, case, dev)
            for (idx, vb, vl), (c, d) in zip(case, res):
                G = oracle.unpack_subset(w.packed, w.n, w.m, idx, vb, vl)
                oc, od, _ = oracle.ibs_triangle_from_codes(G)
                assert (c == oc).all(), f"n={idx.size} window={vb}+{vl}"
                assert_dist_close(d, od)
    finally:
        ibs.ibs_shutdown(ctx)


def _random_pool(n, m, seed):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(0, 256, (m, (n + 3) // 4), dtype=torch.uint8, device="cuda", generator=g)


def _subset_args(pool_n, n, vb, vl, seed, dist=True):
    import torch
    idx = np.sort(np.random.default_rng(seed).choice(pool_n, size=n, replace=False)).astype(np.int64)
    P = n * (n + 1) // 2
    return [(torch.from_numpy(idx).cuda(), vb, vl, torch.full((P, 4), -7, dtype=torch.int32, device="cuda"),
             torch.empty(P, dtype=torch.float64, device="cuda") if dist else None)]


def test_plans_share_the_regrouped_pool():
    """Batches of other sizes of one pool: each plan keeps planes and parts of
    its own, but not another copy of the pool (0.8 GB here)."""
    import torch
    from paper_1410_4803_gb300 import ibs
    pool_n, m = 4096, 800_000
    pool = _random_pool(pool_n, m, 1)
    calls = [_subset_args(pool_n, n, 0, m, n) for n in (1025, 1026, 1027)]
    ctx = ibs.ibs_init(0, flags=ibs.IBS_KERNEL_TC | ibs.IBS_TC_FP4)
    try:
        held = []
        for subs in calls:
            torch.cuda.synchronize()
            before = torch.cuda.mem_get_info()[0]
            ibs.ibs_compute_batch(ctx, pool, pool_n, m, subs)
            ibs.ibs_synchronize(ctx)
            held.append(before - torch.cuda.mem_get_info()[0])
        planes = 17 * 64 * 2 * m
        assert held[0] > planes + 0.8e9  # the pool is regrouped
        assert max(held[1:]) < planes + 0.5e9, held
    finally:
        ibs.ibs_shutdown(ctx)


def test_batches_on_two_streams():
    """Two plans whose pools are regrouped, back to back on two streams: the
    results of each alone."""
    import torch
    from paper_1410_4803_gb300 import ibs
    pool_n, m = 2048, 60_000
    pool = _random_pool(pool_n, m, 2)
    calls = [_subset_args(pool_n, 900, 0, 30_000, 1), _subset_args(pool_n, 700, 29_001, 30_999, 2)]
    ctx = ibs.ibs_init(0, flags=ibs.IBS_KERNEL_TC | ibs.IBS_TC_FP4)
    try:
        want = []
        for subs in calls:
            ibs.ibs_compute_batch(ctx, pool, pool_n, m, subs)
            ibs.ibs_synchronize(ctx)
            want.append(subs[0][3].clone())
        streams = [torch.cuda.Stream() for _ in calls]
        for _ in range(5):
            for subs in calls:
                subs[0][3].fill_(-7)
            torch.cuda.synchronize()
            for subs, st in zip(calls, streams):
                ibs.ibs_compute_batch(ctx, pool, pool_n, m, subs, stream=st)
            torch.cuda.synchronize()
            for subs, w in zip(calls, want):
                assert torch.equal(subs[0][3], w)
    finally:
        ibs.ibs_shutdown(ctx)


def test_tune_file_and_the_sweep_kernel(tmp_path):
    """The sweep kernel's batches are not timed: an entry of another policy does
    not keep a batch off it, and it leaves no entry that a context which cannot
    take it (a workspace limit) would follow unmeasured."""
    import json
    from paper_1410_4803_gb300 import ibs
    pool_n, m = 600, 3000
    pool = _random_pool(pool_n, m, 3)
    subs = [_subset_args(pool_n, n, 0, vl, n)[0] for n, vl in ((300, 3000), (150, 2000), (90, 2500), (200, 900))]
    path = tmp_path / "tune.jsonl"

    def run(**kw):
        """Kernel launches of the batch on a new context, and the file's entries after it."""
        for s in subs:
            s[3].fill_(-7)
        ctx = ibs.ibs_init(0, flags=ibs.IBS_KERNEL_TC | ibs.IBS_TC_FP4, autotune_cache_path=str(path), **kw)
        try:
            ibs.ibs_compute_batch(ctx, pool, pool_n, m, subs)
            ibs.ibs_synchronize(ctx)
            launches = ibs.ibs_last_launch_info(ctx)["launches"]
        finally:
            ibs.ibs_shutdown(ctx)
        return launches, [json.loads(x) for x in path.read_text().splitlines()]

    launches, entries = run()
    assert launches <= 3  # gather, sweeps, sums
    want = [s[3].clone() for s in subs]
    assert all(e["ms"] == 0 for e in entries)
    _, entries = run(workspace_bytes=256 << 20)
    timed = [e for e in entries if e["ms"] > 0]
    assert len(timed) == 1
    for s, w in zip(subs, want):
        assert (s[3] == w).all()
    # the entry of another policy
    path.write_text(json.dumps(dict(timed[0], split=0)) + "\n")
    launches, entries = run()
    assert launches <= 3
    assert [e for e in entries if e["ms"] > 0] == [dict(timed[0], split=0)]
    # an untimed entry under a timed policy's key is measured anew
    path.write_text(json.dumps(dict(timed[0], ms=0.0, split=2)) + "\n")
    _, entries = run(workspace_bytes=256 << 20)
    assert len([e for e in entries if e["ms"] > 0]) == 1


@pytest.mark.parametrize("m,dist,timed", [(9_999, False, True), (10_000, False, False), (300, True, False)])
def test_batch_of_counts_alone(tmp_path, m, dist, timed):
    """Batches without distances: either side of the mean marker count at which
    they go to the timed policies; the plan of the same shapes with distances is
    another."""
    import json
    import torch
    from paper_1410_4803_gb300 import ibs
    pool_n = 300
    pool = _random_pool(pool_n, m, 5)
    subs = [_subset_args(pool_n, n, 0, m, n, dist=False)[0] for n in (140, 150, 90)]
    with_dist = [s[:4] + (torch.empty(s[3].shape[0], dtype=torch.float64, device="cuda"),) for s in subs]
    path = tmp_path / "tune.jsonl"
    ctx = ibs.ibs_init(0, flags=ibs.IBS_KERNEL_TC | ibs.IBS_TC_FP4, autotune_cache_path=str(path))
    try:
        for use in ((with_dist, with_dist) if dist else (subs, with_dist, subs)):
            for s in subs:
                s[3].fill_(-7)
            ibs.ibs_compute_batch(ctx, pool, pool_n, m, use)
            ibs.ibs_synchronize(ctx)
            for s in subs:
                G = oracle.unpack_subset(pool.cpu().numpy(), pool_n, m, s[0].cpu().numpy(), 0, m)
                assert (s[3].cpu().numpy() == oracle.ibs_triangle_from_codes(G)[0]).all()
    finally:
        ibs.ibs_shutdown(ctx)
    assert any(json.loads(x)["ms"] > 0 for x in path.read_text().splitlines()) == timed


@pytest.mark.parametrize("n,m,timed", [(16, 12_000, False), (16, 12_001, True), (100, 32_000, False),
                                       (100, 32_001, True), (128, 39_841, True), (129, 39_841, False)])
def test_lone_narrow_subset(tmp_path, n, m, timed):
    """Either side of the sizes at which a lone subset of one block of samples
    goes to the timed policies."""
    import json
    from paper_1410_4803_gb300 import ibs
    pool_n = 150
    pool = _random_pool(pool_n, m, n)
    subs = _subset_args(pool_n, n, 0, m, n)
    path = tmp_path / "tune.jsonl"
    ctx = ibs.ibs_init(0, flags=ibs.IBS_KERNEL_TC | ibs.IBS_TC_FP4, autotune_cache_path=str(path))
    try:
        for _ in range(2):
            subs[0][3].fill_(-7)
            ibs.ibs_compute_batch(ctx, pool, pool_n, m, subs)
            ibs.ibs_synchronize(ctx)
            G = oracle.unpack_subset(pool.cpu().numpy(), pool_n, m, subs[0][0].cpu().numpy(), 0, m)
            assert (subs[0][3].cpu().numpy() == oracle.ibs_triangle_from_codes(G)[0]).all()
    finally:
        ibs.ibs_shutdown(ctx)
    assert any(json.loads(x)["ms"] > 0 for x in path.read_text().splitlines()) == timed


POLICY5_CHILD = r"""
import sys
import numpy as np
sys.path.insert(0, {tests!r}); sys.path.insert(0, {root!r})
import torch
import oracle
from helpers import assert_dist_close
from test_gpu_batch import _flags, _make_subsets, _run_batch
from paper_1410_4803_gb300 import ibs, synth
w = synth.batch_pool(pool_n=1500, pool_m=30000, seed=11)
subs = _make_subsets(np.random.default_rng(9), w.n, w.m)
ctx = ibs.ibs_init(0, flags=_flags(ibs, "IBS_KERNEL_TC|IBS_TC_FP4"))
dev = torch.from_numpy(w.packed).cuda()
first = _run_batch(ctx, w, subs, dev)
second = _run_batch(ctx, w, subs, dev)
assert ibs.ibs_batch_plan_info(ctx)["split_policy"] == 5
launches = ibs.ibs_last_launch_info(ctx)["launches"]
for (idx, vb, vl), (c1, d1), (c2, d2) in zip(subs, first, second):
    G = oracle.unpack_subset(w.packed, w.n, w.m, idx, vb, vl)
    oc, od, _ = oracle.ibs_triangle_from_codes(G)
    assert (c1 == oc).all(), f"n={{idx.size}} window={{vb}}+{{vl}}"
    assert (c2 == oc).all()
    assert_dist_close(d1, od)
    np.testing.assert_array_equal(d1, d2)
ibs.ibs_shutdown(ctx)
print("ok", launches)
"""


def test_batch_policy5_fused_gather():
    """Policy 5 with the two-SM kernel forced on for every subset of two or
    more blocks (IBS_TC_PAIR=1, read once per process: a child): the order
    mixes two-SM subsets, whose epilogue warps gather the planes of the
    subsets after them, and one-SM subsets (n <= 128), which the preceding
    two-SM launch gathers; the first subset gets a gather launch of its own.
    Counts equal the oracle for all twelve subsets, twice (graph replay)."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    code = POLICY5_CHILD.format(tests=os.path.join(root, "tests"), root=root)
    env = dict(os.environ, IBS_TC_PAIR="1", IBS_BATCH_POLICY="5")
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "ok" in r.stdout, r.stdout
