"""Two changes of route that depend on sizes not seen in the rows: a key with
more records than a block groups, in a partition that holds them, and the
largest bound of records for which a search does not wait for their count."""
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


def test_key_past_a_blocks_list(xtn):
    """A plan's regions are for every deletion subset: 11,000 records each in 256
    partitions, where sequences of five runs give 2,300 or so.  6,500 copies of
    a run of one residue (two variants) fit as well, but a block groups 6,144."""
    n, copies, d = 100_000, 6_500, 1
    rng = np.random.default_rng(4)
    ends = np.sort(rng.integers(1, 25, (n, 4)), axis=1)
    run = (np.arange(25)[None, :, None] >= ends[:, None, :]).sum(axis=2)
    m = np.take_along_axis(rng.choice(gen.AA_BYTES, (n, 5)), run, axis=1)
    m[rng.choice(n, copies, replace=False)] = ord("W")
    off = np.arange(n + 1, dtype=np.int64) * 25
    ds, do = torch.from_numpy(m.reshape(-1).copy()).cuda(), torch.from_numpy(off).cuda()
    cap = copies * copies // 2 + n
    plan = xtn.Plan(off, d, pair_capacity=3 * cap)
    plan.run(ds)
    got = plan.result(cap=cap, like=ds)
    stats = plan.stats()
    # no partition runs over, so what the global grouping got came from lists
    assert 1.5 * stats["records"] / 256 + copies < plan.info()["record_capacity"] / 256
    assert 2 <= stats["groups"] < 2_000
    plan.free()
    old = xtn.tune_get(xtn.XTN_TUNE_GROUPING)
    xtn.tune_set(xtn.XTN_TUNE_GROUPING, 1)
    try:
        want = xtn.search_self(ds, do, d, cap=cap)
    finally:
        xtn.tune_set(xtn.XTN_TUNE_GROUPING, old)
    assert len(want) >= copies * (copies - 1) // 2 and torch.equal(got, want)


def test_front_without_a_wait(xtn):
    """326 records a sequence of 25 at d = 2 at most: 12,865 of them make fewer
    than 2^22, 12,866 more."""
    waits = []
    for n in (12_865, 12_866):
        seqs, off = gen.generate(n, n, 0.3, 0.02)
        ds, do = torch.from_numpy(seqs).cuda(), torch.from_numpy(off).cuda()
        want = oracle.symdel_self_sharded(seqs, off, 2)
        xtn.search_self(ds, do, 2, cap=len(want))
        xtn.profile_report()
        xtn.profile_enable(True)
        got = xtn.search_self(ds, do, 2, cap=len(want))
        xtn.profile_enable(False)
        waits.append(xtn.profile_report()["host_stream_wait"][0])
        assert np.array_equal(got.cpu().numpy().astype(np.uint32), want)
    assert waits[1] == waits[0] + 1
