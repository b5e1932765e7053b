"""Two levels of partitions (more than 655 M records, or a plan's bound of
them): coarse and fine partitions that run over, one-shot, in passes and
planned, and word indices past 32 bits, against the CPU oracle or the grouping
by global sorting."""
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
    torch.cuda.empty_cache()
    pkg.scratch_trim()
    yield pkg
    torch.cuda.empty_cache()
    pkg.scratch_trim()


def _kernels(xtn, call):
    xtn.profile_report()
    xtn.profile_enable(True)
    try:
        out = call()
    finally:
        xtn.profile_enable(False)
    return out, xtn.profile_report()


def _by_sorting(xtn, call):
    old = xtn.tune_get(xtn.XTN_TUNE_GROUPING)
    xtn.tune_set(xtn.XTN_TUNE_GROUPING, 1)
    try:
        return call()
    finally:
        xtn.tune_set(xtn.XTN_TUNE_GROUPING, old)


def _few_runs(n, seed):
    """n sequences of 25 residues in five runs (about 56 of their 2,626
    deletion subsets at d = 3 are distinct strings), some repeated."""
    rng = np.random.default_rng(seed)
    ends = np.sort(rng.integers(1, 25, (n, 4)), axis=1)
    letters = rng.choice(gen.AA_BYTES, (n, 5))
    run = (np.arange(25)[None, :, None] >= ends[:, None, :]).sum(axis=2)
    m = np.take_along_axis(letters, run, axis=1)
    m[rng.integers(0, n, n // 50)] = m[rng.integers(0, n, n // 50)]
    return np.ascontiguousarray(m).reshape(-1), np.arange(n + 1, dtype=np.int64) * 25


# 661.8 M and 4,290.9 M of 2,626 a sequence: the second's regions together are
# past 2^32 words on both levels
@pytest.mark.parametrize("n", [252_001, 1_634_001])
def test_plan_with_two_levels(xtn, n):
    seqs, off = _few_runs(n, n)
    ds, do = torch.from_numpy(seqs).cuda(), torch.from_numpy(off).cuda()
    plan = xtn.Plan(off, 3, pair_capacity=100 * n)
    assert plan.info()["record_capacity"] == 2626 * n
    _, kernels = _kernels(xtn, lambda: plan.run(ds))
    assert kernels["k_split"][0] == 1
    got = plan.result(cap=8 * n, like=ds)
    plan.run(ds)  # once more over the first run's buffers
    assert torch.equal(plan.result(cap=8 * n, like=ds), got)
    plan.free()
    want = _by_sorting(xtn, lambda: xtn.search_self(ds, do, 3, cap=8 * n))
    assert len(want) > n // 100 and torch.equal(got, want)
    if n < 300_000:
        assert np.array_equal(got.cpu().numpy().astype(np.uint32),
                              oracle.symdel_self_sharded(seqs, off, 3))


def test_partitions_of_either_level_run_over(xtn):
    """About 690 M records: a coarse region has room for 9,400 records past its
    mean, a fine one for 1,800.  A run of one residue has two variants at
    d = 1, so 16,000 copies of one overflow two coarse partitions and 6,000 of
    another two fine ones."""
    n, L = 45_000_000, 15
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    letters = torch.from_numpy(gen.AA_BYTES.copy()).cuda()
    ds = torch.empty(n, L, dtype=torch.uint8, device="cuda")
    for k in range(L):
        ds[:, k] = letters[torch.randint(0, 20, (n,), generator=g, device="cuda")]
    at = torch.randperm(n, generator=g, device="cuda")[:22_000]
    ds[at[:16_000]] = ord("A")
    ds[at[16_000:]] = ord("C")
    ds = ds.reshape(-1)
    do = torch.arange(n + 1, device="cuda", dtype=torch.int64) * L
    cap = 150_000_000
    got, kernels = _kernels(xtn, lambda: xtn.search_self(ds, do, 1, cap=cap))
    assert kernels["k_split"][0] == 1 and kernels["k_emit_pairs"][0] == 1
    assert len(got) >= 16_000 * 15_999 // 2 + 6_000 * 5_999 // 2
    want = _by_sorting(xtn, lambda: xtn.search_self(ds, do, 1, cap=cap))
    assert torch.equal(got, want)
    del want
    (rows, passes), kernels = _kernels(xtn, lambda: xtn.search_self_streaming(
        ds, do, 1, max_pass_records=800_000_000, cap=cap))
    assert passes == 1 and kernels["k_split"][0] == 1
    assert torch.equal(rows, got)


def _subsets_d3(m):
    """Distinct strings after at most three deletions, per row of m (their
    number goes by the runs of equal residues: R, two or longer, three or
    longer)."""
    eq = m[:, 1:] == m[:, :-1]
    start = torch.ones_like(m, dtype=torch.bool)
    start[:, 1:] = ~eq
    long2 = start[:, :-1] & eq
    long3 = long2[:, :-1] & eq[:, 1:]
    R, D, T = (x.sum(1).long() for x in (start, long2, long3))
    return (1 + R + R * (R - 1) // 2 + D + R * (R - 1) * (R - 2) // 6 + D * (R - 1) + T)


def test_word_indices_past_32_bits(xtn):
    """4,285 to 4,294 M records at once: in one pass (the regions together are
    past 2^32 words there, too, and the records come through k_partition) and in
    one search, against passes of a quarter."""
    n, L = 2_100_000, 25
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    letters = torch.from_numpy(gen.AA_BYTES.copy()).cuda()
    m = letters[torch.randint(0, 20, (n, L), generator=g, device="cuda")]
    src = torch.randint(0, n // 2, (n // 40,), generator=g, device="cuda")
    at = n // 2 + torch.randperm(n // 2, generator=g, device="cuda")[:n // 40]
    m[at] = m[src]  # copies, then one to three residues of most of them changed
    for _ in range(3):
        m[at, torch.randint(0, L, (n // 40,), generator=g, device="cuda")] = \
            letters[torch.randint(0, 20, (n // 40,), generator=g, device="cuda")]
    limit = (1 << 32) - (1 << 20)
    upto = torch.cumsum(_subsets_d3(m), 0)
    n = int((upto < limit - 1_000_000).sum())
    total = int(upto[n - 1])
    assert 4_285_000_000 < total < limit
    ds = m[:n].reshape(-1).contiguous()
    do = torch.arange(n + 1, device="cuda", dtype=torch.int64) * L
    want, passes = xtn.search_self_streaming(ds, do, 3, max_pass_records=1 << 30)
    assert passes > 3 and len(want) > n // 100
    (rows, passes), kernels = _kernels(xtn, lambda: xtn.search_self_streaming(
        ds, do, 3, max_pass_records=limit))
    assert passes == 1 and kernels["k_split"][0] == 1
    assert torch.equal(rows, want)
    got, kernels = _kernels(xtn, lambda: xtn.search_self(ds, do, 3))
    assert kernels["k_split"][0] == 1 and "k_expand_bins" not in kernels
    assert torch.equal(got, want)
