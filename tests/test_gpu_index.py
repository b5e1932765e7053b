"""An index built out of partitions, against one built by sorting (grouping
mode 1) and the CPU oracle: one record, directory ranges that are sorted by a
warp and by a block, one beyond what a block holds, partitions that run over,
expansions split and in one kernel, partitions placed in several fills."""
import numpy as np
import pytest

import cdr3_synth as gen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _rows(x):
    return x.cpu().numpy().astype(np.uint32)


@pytest.mark.parametrize("n,d,copies", [
    (1, 0, []), (1, 3, []), (300, 2, [33, 34, 1025]), (3000, 1, [5000]),
    (2000, 1, [30_000]),                  # one range beyond a block's stage
    (100, 0, [20_000]), (9_000, 3, [40]),
    (70_000, 2, [600]),                   # one kernel expands into partitions
    (420_000, 2, [50])])                  # more than one fill of a partition
def test_index_build(n, d, copies):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2403_09010_gb300 as xtn
    xtn.build()
    rng = np.random.default_rng(n + d)
    strs = gen.to_strings(*gen.generate(n, n, 0.3, 0.02))
    for k, c in enumerate(copies):
        strs += ["CASS" + "LGTDY"[k:] + "TQYF"] * c
    strs += ["", "A" * 25][: len(strs) - 1]
    seqs, off = gen.from_strings([strs[i] for i in rng.permutation(len(strs))])
    q, qo = gen.from_strings([strs[i] for i in rng.integers(0, len(strs), 50)] + ["A", ""])
    ds, do, dq, dqo = [torch.from_numpy(a).cuda() for a in (seqs, off, q, qo)]
    old = xtn.tune_get(xtn.XTN_TUNE_GROUPING)
    got = {}
    for mode in (0, 1):
        xtn.tune_set(xtn.XTN_TUNE_GROUPING, mode)
        try:
            idx = xtn.index_build(ds, do, d)
        finally:
            xtn.tune_set(xtn.XTN_TUNE_GROUPING, old)
        got[mode] = (_rows(xtn.search_query(idx, dq, dqo, cap=4_000_000)),
                     idx.scratch_bytes(qo) if mode == 0 else None)
        idx.free()
    assert np.array_equal(got[0][0], got[1][0])
    if n <= 9_000:
        assert np.array_equal(got[0][0], oracle.bruteforce_query(seqs, off, q, qo, d, threads=0))
