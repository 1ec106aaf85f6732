"""Parity of vardrop_select with the oracle: every output bit-exact (integer work)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2501_14183_b200 import binding as vd
from paper_2501_14183_b200 import inputs

pytestmark = pytest.mark.gpu


def run_select(keys, gs, rate, seed, step):
    keys = np.atleast_2d(keys)
    S, N = keys.shape
    cfg = vd.SelectCfg(S, N, gs, rate, seed, step)
    kd = torch.from_numpy(keys.view(np.int64)).cuda()
    out = vd.alloc_select_outputs(cfg)
    ws = vd.alloc_ws(vd.vardrop_select_workspace_bytes(cfg))
    vd.vardrop_select(kd, cfg, out["group_id"], out["group_offsets"], out["members"], out["n_groups"], out["sel_idx"],
                      out["n_sel"], out["inv_idx"], ws)
    torch.cuda.synchronize()
    assert vd.ws_status(ws) == vd.OK
    return {k: v.cpu().numpy() for k, v in out.items()}


def check(keys, gs, rate, seed, step):
    want = oracle.select(keys, gs, rate, seed, step)
    got = run_select(keys, gs, rate, seed, step)
    for name in ("n_groups", "n_sel", "group_id", "group_offsets", "members", "sel_idx", "inv_idx"):
        assert np.array_equal(got[name], want[name]), name
    return got


@pytest.mark.parametrize("N,G", [(1, 1), (2, 2), (21, 4), (127, 9), (128, 128), (129, 1), (257, 30), (321, 40), (862, 60),
                                 (1000, 1000), (3000, 7), (8192, 512)])
@pytest.mark.parametrize("gs,rate", [(10, 1.0), (0, 0.2), (3, 0.5)])
def test_select_parity(N, G, gs, rate):
    keys = inputs.make_keys(N, G, k=4, f_hi=85, seed=N + G)
    check(keys, gs, rate, seed=0xC0FFEE1234567, step=N % 7)


def test_select_degenerate_groups():
    same = np.full(2000, (5 << 24) | (9 << 12) | 2, dtype=np.uint64)
    got = check(same, 10, 1.0, seed=1, step=0)
    assert got["n_groups"][0] == 1 and got["n_sel"][0] == 10
    distinct = np.arange(1, 1501, dtype=np.uint64)[np.random.default_rng(0).permutation(1500)]
    got = check(distinct, 10, 1.0, seed=1, step=0)
    assert got["n_groups"][0] == 1500 and got["n_sel"][0] == 1500
    check(np.full(300, 0xFFFFFFFFFFFFFFF, dtype=np.uint64), 0, 0.1, seed=3, step=9)     # 60-bit keys (k = 5)


def test_select_group_sizes_around_the_counting_limit():
    """Members are ranked by counting inside groups of up to 64 and by buckets of their priorities in longer ones: both sides of it."""
    rng = np.random.default_rng(11)
    for sizes in ([64, 64, 64], [65, 64, 64], [64, 1, 63, 2], [300, 5, 5, 5], [1] * 40 + [64]):
        keys = np.concatenate([np.full(n, 100 + 7 * i, dtype=np.uint64) for i, n in enumerate(sizes)])
        keys = keys[rng.permutation(len(keys))]
        for gs, rate in ((10, 1.0), (0, 0.3)):
            check(keys, gs, rate, seed=99, step=4)


@pytest.mark.parametrize("N,G", [(64, 64), (65, 63), (255, 182), (256, 183), (512, 256), (513, 159), (513, 257), (862, 160), (1024, 160), (1000, 161), (1024, 362), (1000, 363),
                                 (129, 129), (200, 160), (256, 161), (512, 257), (513, 352), (1024, 353), (1025, 360), (2048, 360), (1500, 361), (2048, 512), (1500, 513), (2048, 16), (1100, 9), (513, 1), (862, 2), (1024, 3), (2048, 1)])
def test_select_group_counts_around_the_counting_limit(N, G):
    """Few and many distinct keys in every size range: up to 128 variates all of them have entries in the hash table, up to 256, 512 and 1024 as long as they are
    no more than 160, 256 and 352 (then they are sorted), above that all pairs are compared; one key is all ones, the mark of a free slot of the table and
    not a number where keys are compared as doubles."""
    rng = np.random.default_rng(N * 7 + G)
    values = np.unique(rng.integers(1, 1 << 60, 2 * G, dtype=np.uint64))[:G]
    values[G // 2] = np.uint64(0xFFFFFFFFFFFFFFFF)
    keys = values[np.concatenate([np.arange(G), rng.integers(0, G, N - G)])] if N > G else values.copy()
    keys = keys[rng.permutation(N)]
    check(np.stack([keys, keys[::-1]]), 0, 0.3, seed=N + G, step=2)


@pytest.mark.parametrize("sizes", [[128] * 5, [129, 128, 128, 128, 1], [300, 213], [1, 1, 1000], [128, 600, 128, 100, 1], [2000, 48], [700, 700, 648]])
def test_select_group_lengths_around_the_counting_limit(sizes):
    """Long groups, whose sampling ranks come from buckets of their priorities, alone and among others, on one CTA and over several."""
    keys = np.concatenate([np.full(n, 7919 * (i + 3) % 1000, dtype=np.uint64) for i, n in enumerate(sizes)])
    keys = keys[np.random.default_rng(len(keys)).permutation(len(keys))]
    for gs, rate in ((10, 1.0), (0, 0.3), (0, 1.0), (150, 0.9)):
        check(np.stack([keys, keys[::-1]]), gs, rate, seed=17, step=3)


@pytest.mark.parametrize("N,size", [(60, 60), (64, 64), (65, 65), (500, 64), (862, 60), (1000, 300), (1024, 700), (1025, 64), (1500, 1500), (2000, 60), (3000, 700)])
def test_select_equal_priorities_rank_by_place(N, size):
    """Members 13 and 36 of the first group draw the same 32-bit priority under this seed and step (found by search): with the quota
    between them the earlier one is kept.  Short groups, which count their ranks, and long ones, in every size range."""
    seed, step = 77, 3689518
    rank = {60: 21, 64: 23, 65: 23, 300: 113, 700: 256, 1500: 548}[size]       # members of lower priority
    keys = np.concatenate([np.full(size, 5, dtype=np.uint64), 6 + np.arange(N - size, dtype=np.uint64) // 20])
    keys = keys[np.random.default_rng(N).permutation(N)]
    for gs in (rank, rank + 1, rank + 2):
        check(keys, gs, 1.0, seed=seed, step=step)


@pytest.mark.parametrize("N", [2, 63, 64, 65, 128, 129, 256, 257, 512, 513, 1023, 1024, 1025, 1026, 2047, 2048, 2049, 2368, 2369, 4096, 4097, 4736, 4737, 8191, 8192, 8193])
def test_select_group_shapes_at_the_size_limits(N):
    """Both sides of the sizes at which a path, its tables or a CTA's share change: few and many groups, some of 64 and 65 members (ranks counted, and
    found by buckets), long ones that reach over several CTAs' positions, all distinct."""
    rng = np.random.default_rng(N)
    for sizes in ([N], [1] * N, [64, 65] * (N // 129) + [N % 129], [N // 2, N // 3, N - N // 2 - N // 3], [9] * (N // 9) + [N % 9]):
        sizes = [n for n in sizes if n > 0]
        values = rng.permutation(np.unique(rng.integers(0, 1 << 56, 2 * len(sizes), dtype=np.uint64)))[:len(sizes)]
        keys = np.repeat(values, sizes)[rng.permutation(N)]
        check(keys, 0, 0.3, seed=N, step=1)
        check(np.stack([keys, keys[::-1]]), 40, 1.0, seed=N, step=2)


@pytest.mark.parametrize("S,N,G", [(18, 1025, 100), (9, 1500, 360), (8, 2048, 361), (6, 2000, 3), (6, 2048, 2048), (8, 2047, 200), (5, 2048, 1), (5, 2048, 31)])
def test_select_many_rows_of_1025_to_2048(S, N, G):
    """With this many rows one CTA a row takes them, two variates a thread: few and many distinct keys, more than the table takes, long groups."""
    rng = np.random.default_rng(N + G)
    values = rng.permutation(np.unique(rng.integers(0, 1 << 60, 2 * G, dtype=np.uint64)))[:G]
    rows = np.stack([values[np.concatenate([np.arange(G), rng.integers(0, G, N - G)])][rng.permutation(N)] for _ in range(S)])
    check(rows, 0, 0.3, seed=N, step=1)
    check(rows, 12, 1.0, seed=G, step=2)


@pytest.mark.parametrize("S,N,launches", [(1, 1024, 1), (32, 1024, 1), (1, 1025, 2), (4, 1025, 2), (5, 1025, 1), (8, 1500, 1), (4, 2048, 2), (5, 2048, 1), (32, 2048, 1), (1, 2049, 2), (32, 2049, 2)])
def test_select_launches_by_rows(S, N, launches):
    """From 1025 to 2048 variates two launches as long as they take no longer than one CTA a row does with few groups."""
    keys = np.stack([inputs.make_keys(N, 40, k=4, f_hi=169, seed=s) for s in range(S)])
    before = vd.vardrop_launch_count()
    check(keys, 0, 0.2, seed=N, step=1)
    assert vd.vardrop_launch_count() == before + launches


def test_select_long_rows():
    """Rows beyond the cluster's: grouping with its working arrays in shared memory (up to 18432 variates), at that
    limit, and on the global arrays beyond it; several rows at once; one group only and all-distinct keys."""
    for N, G in ((18432, 700), (18433, 50), (24000, 3000)):
        check(inputs.make_keys(N, G, k=4, f_hi=169, seed=N), 10, 1.0, seed=42, step=2)
    rows = np.stack([inputs.make_keys(2500, 30 + 40 * s, k=3, f_hi=49, seed=90 + s) for s in range(3)])
    check(rows, 0, 0.25, seed=7, step=1)
    rows = np.stack([inputs.make_keys(19000, 100 + 900 * s, k=4, f_hi=169, seed=190 + s) for s in range(2)])
    check(rows, 4, 0.5, seed=8, step=6)
    got = check(np.full(5000, 77, dtype=np.uint64), 0, 0.1, seed=3, step=0)
    assert got["n_groups"][0] == 1 and got["n_sel"][0] == 500
    distinct = np.arange(1, 4097, dtype=np.uint64)[np.random.default_rng(1).permutation(4096)]
    got = check(distinct, 10, 1.0, seed=1, step=0)
    assert got["n_groups"][0] == 4096 and got["n_sel"][0] == 4096


def test_select_middle_rows():
    """Rows of 2049 .. 8192 variates (all pairs and a cluster): ragged sizes, keys that differ in all 64 bits or in a single one, one group, two groups
    of very different size, many equal groups of 512, 20 and 2 members, several rows at once."""
    rng = np.random.default_rng(5)
    wide = rng.integers(0, 2**63, size=5000, dtype=np.uint64) * np.uint64(2) + rng.integers(0, 2, size=5000, dtype=np.uint64)
    wide[rng.integers(0, 5000, size=700)] = wide[0]                        # one longer group among distinct keys
    wide[1] = np.uint64(0xFFFFFFFFFFFFFFFF)
    wide[2] = np.uint64(0)
    check(wide, 10, 1.0, seed=12, step=3)
    check(wide, 0, 0.3, seed=12, step=4)
    one_bit = (rng.integers(0, 2, size=8191, dtype=np.uint64) << np.uint64(63)) | np.uint64(0x123)
    got = check(one_bit, 0, 0.01, seed=2, step=0)
    assert got["n_groups"][0] == 2
    for N in (2049, 3073, 8191, 8192):
        for sizes in ([N], [N - 1, 1], [512] * (N // 512) + [N % 512], [20] * (N // 20) + [N % 20], [2] * (N // 2) + [N % 2]):
            sizes = [n for n in sizes if n > 0]
            keys = np.concatenate([np.full(n, (i * 0x9E3779B97F4A7C15) % 2**48, dtype=np.uint64) for i, n in enumerate(sizes)])
            keys = keys[rng.permutation(len(keys))]
            check(keys, 7, 0.4, seed=N, step=len(sizes) % 5)
    rows = np.stack([inputs.make_keys(6000, 10 + 700 * s, k=5, f_hi=361, seed=60 + s) for s in range(4)])
    check(rows, 0, 0.1, seed=31, step=2)


def test_select_random_configurations():
    """Seeded random draws of (N, rows, groups, gs, rate, k) on both sides of every size limit of the kernels
    (1024: one-CTA path; 8192: all pairs and a cluster; 18432: grouping in shared memory; 65536: the largest N)."""
    rng = np.random.default_rng(123)
    for it in range(24):
        N = int(rng.choice([63, 64, 65, 700, 2047, 2048, 2049, 4096, 8192, 18432, 18433, 30000, 65536]))
        S = int(rng.choice([1, 1, 2, 3])) if N <= 20000 else 1
        G = int(rng.integers(1, max(2, N // int(rng.choice([1, 2, 8, 50, 400])))))
        gs = int(rng.choice([0, 1, 3, 10, 100]))
        rate = float(rng.choice([0.05, 0.2, 0.5, 1.0]))
        k = int(rng.choice([3, 4, 5]))
        rows = np.stack([inputs.make_keys(N, G, k=k, f_hi=int(rng.choice([25, 49, 169, 361])), seed=1000 * it + s) for s in range(S)])
        check(rows, gs, rate, seed=int(rng.integers(0, 2**62)), step=int(rng.integers(0, 1000)))


def test_select_multiple_scopes():
    rows = np.stack([inputs.make_keys(500, 20 + s, k=3, f_hi=25, seed=s) for s in range(5)])
    got = check(rows, 5, 1.0, seed=77, step=3)
    assert len(set(got["n_sel"].tolist())) > 1


def test_select_paper_hyperparameters():
    # (k, gs) of Appendix E on keys hashed from the synthetic workloads
    for name, gs in (("elec", 10), ("traffic", 10), ("tiny", 5)):
        w = inputs.WORKLOADS[name]
        keys, _, _ = oracle.hash(inputs.make_windows(w, B=4), w.k)
        got = check(keys, gs, 1.0, seed=20250114, step=1)
        sizes = np.diff(got["group_offsets"][0][: got["n_groups"][0] + 1])
        assert got["n_sel"][0] == np.minimum(sizes, gs).sum()           # Eq. 1 summed over groups


def test_select_reproducible_and_step_dependent():
    keys = inputs.make_keys(862, 60, k=3, f_hi=25, seed=2)
    a = run_select(keys, 0, 0.2, seed=5, step=10)
    b = run_select(keys, 0, 0.2, seed=5, step=10)
    c = run_select(keys, 0, 0.2, seed=5, step=11)
    assert np.array_equal(a["sel_idx"], b["sel_idx"])
    assert not np.array_equal(a["sel_idx"], c["sel_idx"])
    assert a["n_sel"][0] == c["n_sel"][0]


def test_select_argument_errors():
    keys = torch.zeros((1, 8), dtype=torch.int64, device="cuda")
    cfg = vd.SelectCfg(1, 8, 0, 0.5, 1, 0)
    out = vd.alloc_select_outputs(cfg)
    args = (out["group_id"], out["group_offsets"], out["members"], out["n_groups"], out["sel_idx"], out["n_sel"], out["inv_idx"])
    small = vd.alloc_ws(256)
    with pytest.raises(vd.VardropError) as e:
        vd.vardrop_select(keys, cfg, *args, small[:128])
    assert e.value.status == vd.ERR_WORKSPACE
    ws = vd.alloc_ws(vd.vardrop_select_workspace_bytes(cfg))
    for bad in (vd.SelectCfg(1, 8, 0, 0.0, 1, 0), vd.SelectCfg(1, 8, 0, 1.5, 1, 0), vd.SelectCfg(1, 0, 0, 0.5, 1, 0), vd.SelectCfg(0, 8, 0, 0.5, 1, 0)):
        with pytest.raises(vd.VardropError) as e:
            vd.vardrop_select(keys, bad, *args, ws)
        assert e.value.status == vd.ERR_INVALID_ARG
