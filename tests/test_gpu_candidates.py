"""Searches with several times more candidates than their first buffer holds."""
import numpy as np
import pytest

import cdr3_synth as gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_candidates_past_the_buffer():
    """Sequences ten times each: 45 candidates for ten records, where the buffer
    is for one in two.  The blocks that have not begun by then leave, so that
    the grouping that starts over is not paid for twice; a plan counts all."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2403_09010_gb300 as xtn
    xtn.build()
    rng = np.random.default_rng(2)
    n, copies, L = 60_000, 10, 15
    one = rng.choice(gen.AA_BYTES, (n, L))
    order = rng.permutation(n * copies)
    seqs = np.ascontiguousarray(one[order % n]).reshape(-1)
    off = np.arange(n * copies + 1, dtype=np.int64) * L
    ds, do = torch.from_numpy(seqs).cuda(), torch.from_numpy(off).cuda()
    cap = 50 * n
    got = xtn.search_self(ds, do, 2, cap=cap)
    xtn.profile_report()
    xtn.profile_enable(True)
    again = xtn.search_self(ds, do, 2, cap=cap)
    xtn.profile_enable(False)
    kernels = xtn.profile_report()
    assert torch.equal(again, got)
    # equal sequences (random ones of 15 letters are hardly ever within 2)
    at = np.argsort(order % n, kind="stable").reshape(n, copies)
    at.sort(axis=1)
    i, j = np.triu_indices(copies, 1)
    rows = got.cpu().numpy()
    assert len(rows) >= 45 * n
    same = rows[rows[:, 2] == 0]
    want = np.stack([at[:, i].ravel(), at[:, j].ravel()], 1)
    assert np.array_equal(same[:, :2], want[np.lexsort((want[:, 1], want[:, 0]))])
    assert kernels["k_emit_pairs"][0] == 1  # the search started over
    # both write or count every candidate unless the first one is cut short
    assert kernels["k_group_kept"][1] < 0.5 * kernels["k_emit_pairs"][1]
    plan = xtn.Plan(off, 2, pair_capacity=1 << 20)
    plan.run(ds)
    with pytest.raises(xtn.XtnError) as e:
        plan.result(cap=1, like=ds)
    needed = e.value.needed
    plan.free()
    plan = xtn.Plan(off, 2, pair_capacity=needed)
    plan.run(ds)
    assert torch.equal(plan.result(cap=cap, like=ds), got)
    assert plan.stats()["candidates"] == needed
    plan.free()


def test_candidates_past_the_buffer_of_a_small_search():
    """All partitions of a small search are worked on at once, so blocks have to
    leave in the middle of their list: 1.1 M records, 8 M candidates, room for 1 M."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import oracle
    import paper_2403_09010_gb300 as xtn
    xtn.build()
    rng = np.random.default_rng(3)
    n = 160_000
    m = rng.choice(gen.AA_BYTES, (n, 6))
    m[:, 0], m[:, -1] = ord("C"), ord("F")
    off = np.arange(n + 1, dtype=np.int64) * 6
    seqs = m.reshape(-1).copy()
    ds, do = torch.from_numpy(seqs).cuda(), torch.from_numpy(off).cuda()
    cap = 8_000_000
    got = xtn.search_self(ds, do, 1, cap=cap)
    xtn.profile_report()
    xtn.profile_enable(True)
    again = xtn.search_self(ds, do, 1, cap=cap)
    xtn.profile_enable(False)
    kernels = xtn.profile_report()
    assert torch.equal(again, got)
    assert kernels["k_emit_pairs"][0] == 1  # the search started over
    assert kernels["k_group_kept"][1] < 0.3 * kernels["k_emit_pairs"][1]
    few = 20_000
    want = oracle.symdel_self_sharded(seqs[:6 * few], off[:few + 1], 1)
    part = got[got[:, 1] < few].cpu().numpy().astype(np.uint32)
    assert np.array_equal(part, want)
