"""An index built out of partitions at the ranges its records stand in: sorted
by a warp, by a block, too long for a block, and partitions that run over; each
with the kernels that ran, against one built by sorting."""
import numpy as np
import pytest

import cdr3_synth as gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def xtn():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2403_09010_gb300 as pkg
    pkg.build()
    return pkg


def _sequences(n, copies, seed):
    """n random sequences of 15 residues, copies[k] of them a run of residue k
    (which has d + 1 variants)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    letters = torch.from_numpy(gen.AA_BYTES.copy()).cuda()
    ds = letters[torch.randint(0, 20, (n, 15), generator=g, device="cuda")]
    at = torch.randperm(n, generator=g, device="cuda")
    for k, c in enumerate(copies):
        ds[at[:c]] = letters[k]
        at = at[c:]
    return ds.reshape(-1), torch.arange(n + 1, device="cuda", dtype=torch.int64) * 15


def _build(xtn, ds, do, d, mode):
    old = xtn.tune_get(xtn.XTN_TUNE_GROUPING)
    xtn.tune_set(xtn.XTN_TUNE_GROUPING, mode)
    xtn.profile_report()
    xtn.profile_enable(True)
    try:
        idx = xtn.index_build(ds, do, d)
    finally:
        xtn.profile_enable(False)
        xtn.tune_set(xtn.XTN_TUNE_GROUPING, old)
    return idx, xtn.profile_report()


# (n, d, copies, whether the partitions' records end up sorted globally)
#  100,000, d = 1: 1.5 M records in 256 regions with room for 4,000 past the mean
#  300,000, d = 1: regions of 27,900, so that 12,000 copies overflow one
#  8.4 M, d = 1: 128.5 M records, regions of 95,000, and a block places 19,456
@pytest.mark.parametrize("n,d,copies,by_sorting", [
    (100_000, 1, [33, 600, 1024], False),
    (100_000, 1, [1025, 2_500], False),
    (100_000, 2, [40, 3_000], False),
    (300_000, 1, [12_000, 50], True),
    (8_400_000, 1, [25_000, 40], True),
])
def test_ranges(xtn, n, d, copies, by_sorting):
    ds, do = _sequences(n, copies, n)
    idx, kernels = _build(xtn, ds, do, d, 0)
    assert kernels["k_index_build"][0] == 1
    assert ("k_bucket_sort" in kernels) == by_sorting
    assert kernels["k_encode"][0] == 1  # sorting starts from what is encoded
    ref, kernels = _build(xtn, ds, do, d, 1)
    assert "k_index_build" not in kernels
    runs = ["ACDE"[k] * L for k in range(len(copies)) for L in (13, 14, 15, 16)]
    some = gen.to_strings(ds[:15 * 200].cpu().numpy(), do[:201].cpu().numpy())
    qs, qo = gen.from_strings(runs + some)
    q, o = torch.from_numpy(qs).cuda(), torch.from_numpy(qo).cuda()
    cap = 10 * sum(copies) + 10_000
    got = xtn.search_query(idx, q, o, cap=cap)
    assert len(got) >= sum(copies)
    assert torch.equal(got, xtn.search_query(ref, q, o, cap=cap))
    idx.free()
    ref.free()


@pytest.mark.parametrize("n,d", [(60_000, 1), (100_000, 1), (100_000, 2)])
def test_estimate_of_an_index_that_counts_a_sample(xtn, n, d):
    """Scratch of a first query search, from the distinct keys that a build of a
    million records or more counts in one partition of 16.  Their number there
    is binomial, so the estimate is off by sqrt(15 / keys) <= 0.4% (one sigma);
    a smaller build counts all."""
    ds, do = _sequences(n, [30], n)
    idx, _ = _build(xtn, ds, do, d, 0)
    ref, _ = _build(xtn, ds, do, d, 1)
    qo = np.arange(20_001, dtype=np.int64) * 15
    got, want = idx.scratch_bytes(qo), ref.scratch_bytes(qo)
    if idx.info()["n_records"] < 1 << 20:
        assert got == want
    else:
        assert abs(got - want) <= 0.02 * want
    idx.free()
    ref.free()
