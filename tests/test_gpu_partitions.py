"""The partitioned grouping at the sizes where it can go wrong, against the CPU
oracle: partitions and kept lists that overflow, keys repeated more often than
a block's table holds, partitions of repeats only, one record, every radius
and record path (one-shot, planned, in passes), odd sizes around a tile."""
import numpy as np
import pytest

import cdr3_synth as gen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def xtn():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2403_09010_gb300 as pkg
    pkg.build()
    return pkg


def _rows(x):
    return (x if isinstance(x, np.ndarray) else x.cpu().numpy()).astype(np.uint32)


def _random(rng, n, lo=8, hi=20):
    L = rng.integers(lo, hi + 1, n)
    off = np.zeros(n + 1, np.int64)
    np.cumsum(L, out=off[1:])
    return rng.choice(gen.AA_BYTES, int(off[-1])), off


def _mixed(rng, n_random, copies):
    """n_random random sequences and copies[k] copies of one more each, shuffled."""
    seqs, off = _random(rng, n_random + len(copies))
    strs = gen.to_strings(seqs, off)
    strs = strs[:n_random] + [s for s, c in zip(strs[n_random:], copies) for _ in range(c)]
    return gen.from_strings([strs[i] for i in rng.permutation(len(strs))])


def _check(xtn, seqs, off, d, want, pair_capacity):
    ds = torch.from_numpy(np.ascontiguousarray(seqs)).cuda()
    do = torch.from_numpy(np.ascontiguousarray(off)).cuda()
    assert np.array_equal(_rows(xtn.search_self(ds, do, d)), want)
    plan = xtn.Plan(off, d, pair_capacity=pair_capacity)
    for _ in range(2):  # a plan's second run starts from the first one's buffers
        plan.run(ds)
        assert np.array_equal(_rows(plan.result(cap=len(want) + 1, like=ds)), want)
    plan.free()
    n = off.size - 1
    rows, passes = xtn.search_self_streaming(ds, do, d, max_pass_records=max(1, n * 3))
    assert passes >= 1 and np.array_equal(_rows(rows), want)


@pytest.mark.parametrize("name,d,n_random,copies", [
    ("one", 2, 0, [1]),
    ("two_equal", 2, 0, [2]),
    ("partition_overflow", 1, 200, [300]),          # more copies than a region of ~200 records
    ("partition_overflow_d2", 2, 100, [60, 60, 3]),
    ("dense", 2, 12_000, [2] * 14_000),             # most records repeat
    ("dense_d1", 1, 100, [3] * 4_000),
])
def test_repeats(xtn, name, d, n_random, copies):
    seqs, off = _mixed(np.random.default_rng(len(name) + d), n_random, copies)
    _check(xtn, seqs, off, d, oracle.symdel_self(seqs, off, d), 3_000_000)


def test_key_repeated_more_often_than_a_table_holds(xtn):
    """A group of 6,500 in partitions of 14,000 records: d = 0, one record per
    sequence, so that the candidates stay within their buffer."""
    rng = np.random.default_rng(5)
    c, n = 6_500, 43_000_000
    # distinct random sequences of fixed length, and c copies of one of another
    off = np.arange(n + c + 1, dtype=np.int64) * 10
    seqs = rng.choice(gen.AA_BYTES, 10 * (n + c)).astype(np.uint8)
    at = np.sort(rng.choice(n + c, c, replace=False))
    seqs.reshape(-1, 10)[at] = np.frombuffer(b"CCCCCCCCCC", np.uint8)
    got = xtn.search_self(torch.from_numpy(seqs).cuda(), torch.from_numpy(off).cuda(), 0,
                          cap=30_000_000)
    # every pair of equal sequences, found by sorting the words
    codes = (seqs.reshape(-1, 10) - 64).astype(np.int64) @ (32 ** np.arange(10, dtype=np.int64))
    order = np.argsort(codes, kind="stable")
    start = np.flatnonzero(np.concatenate([[True], np.diff(codes[order]) != 0, [True]]))
    size = np.diff(start)
    parts = [np.stack([at[i], at[j]], 1) for i, j in [np.triu_indices(c, 1)]]
    for s, k in zip(start[:-1][size > 1], size[size > 1]):
        if codes[order[s]] != codes[at[0]]:
            i, j = np.triu_indices(k, 1)
            parts.append(np.stack([order[s + i], order[s + j]], 1))
    want = torch.from_numpy(np.concatenate(parts)).cuda()
    key = want[:, 0] * (n + c) + want[:, 1]
    want = want[torch.argsort(key)]
    assert got.shape[0] == want.shape[0]
    assert torch.equal(got[:, :2].long(), want) and int(got[:, 2].sum()) == 0


@pytest.mark.parametrize("n,d", [(3_001, 3), (9_001, 3), (40_001, 1), (420_001, 1), (70_001, 2)])
def test_expansions(xtn, n, d):
    """Record counts on both sides of the one-kernel expansion's threshold, with
    lengths up to the longest, runs of equal residues and empty sequences."""
    rng = np.random.default_rng(n)
    seqs, off = gen.generate(n, n, 0.3, 0.02)
    strs = gen.to_strings(seqs, off)
    for k in range(0, n, 97):
        strs[k] = "".join(rng.choice(list("AC"), rng.integers(0, 26)))
    seqs, off = gen.from_strings(strs)
    got = xtn.search_self(torch.from_numpy(seqs).cuda(), torch.from_numpy(off).cuda(), d,
                          cap=40 * n)
    assert np.array_equal(_rows(got), oracle.symdel_self_sharded(seqs, off, d))


@pytest.mark.parametrize("fx", [0, 2, 3])
def test_partition_sizes(xtn, fx):
    seqs, off = gen.workload(gen.SELF_1M, 60_000)
    want = oracle.symdel_self_sharded(seqs, off, 2)
    old = xtn.tune_get(xtn.XTN_TUNE_FILTER_SEGMENT)
    xtn.tune_set(xtn.XTN_TUNE_FILTER_SEGMENT, fx)
    try:
        assert np.array_equal(_rows(xtn.search_self(seqs, off, 2)), want)
    finally:
        xtn.tune_set(xtn.XTN_TUNE_FILTER_SEGMENT, old)
