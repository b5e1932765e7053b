"""The paths whose choice depends on how small a call is, at the sizes where
they change over, against the CPU oracle: the last step in one block, the
front without a wait for the record count, one and four rounds of sequences a
block in the encoder, one and eight rows a thread in the TCRdist filter."""
import ctypes

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


def _cuda(*arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


@pytest.mark.parametrize("more", [0, 1, 2])  # 4,095, 4,096 and 4,097 candidates at d = 0
def test_last_step_in_one_block(xtn, more):
    strs = ["CASSLGTDTQYF"] * 91 + ["CASSPGQGAYEQYF"] * 2 * (more > 0) + ["AC"] * 2 * (more > 1)
    strs += ["CASSLGTDTQY", "CASSLGTDTQYFF", "CAASLGTDTQYF", "", "ASSPGQGAYEQYF"]
    strs = [strs[i] for i in np.random.default_rng(more).permutation(len(strs))]
    seqs, off = gen.from_strings(strs)
    ds, do = _cuda(seqs, off)
    for d in range(4):
        want = oracle.bruteforce_self(seqs, off, d)
        assert np.array_equal(_rows(xtn.search_self(ds, do, d, cap=len(want))), want)
        idx = xtn.index_build(ds, do, d)
        qs, qo = gen.from_strings(strs[: 40 + more])
        assert np.array_equal(_rows(xtn.search_query(idx, *_cuda(qs, qo), cap=10_000)),
                              oracle.bruteforce_query(seqs, off, qs, qo, d))
    want = oracle.bruteforce_paired(seqs, off, seqs, off, 1)
    assert np.array_equal(_rows(xtn.search_paired(ds, do, ds, do, 1, cap=len(want))), want)
    rep = np.array([0, 30, 60, len(strs)], np.int64)
    by_rep = oracle.symdel_batched(seqs, off, rep, 1)  # repertoire, rows within it
    want = by_rep[:, 1:].copy()
    want[:, :2] += rep[by_rep[:, :1]].astype(np.uint32)
    assert np.array_equal(_rows(xtn.search_self(ds, do, 1, rep_offsets=rep, cap=len(want))), want)


@pytest.mark.parametrize("n,d", [
    (12_866, 2), (12_867, 2),                       # the record count's bound
    ((1 << 18) - 1, 0), (1 << 18, 1), ((1 << 18) + 1, 1), ((1 << 18) + 1025, 0)])  # rounds
def test_fronts(xtn, n, d):
    seqs, off = gen.generate(n, n, 0.3, 0.02)
    strs = gen.to_strings(seqs, off)
    for k in range(0, n, 1009):
        strs[k] = "ACD"[: k % 4] if k % 2 else "A" * 25
    seqs, off = gen.from_strings(strs)
    want = oracle.symdel_self_sharded(seqs, off, d)
    got = _rows(xtn.search_self(*_cuda(seqs, off), d, cap=len(want)))
    assert np.array_equal(got, want)


@pytest.mark.parametrize("n_rows", [1, 255, 257, 262_144, 262_145])
def test_tcrdist_rows(xtn, n_rows):
    rng = np.random.default_rng(n_rows)
    strs = ["".join(rng.choice(list("ACDEFGHIKLMNPQRSTVWY"), rng.integers(0, 26)))
            for _ in range(300)]
    strs[0], strs[1] = "A" * 25, "Y"
    seqs, off = gen.from_strings(strs)
    rows = np.stack([rng.integers(0, 300, n_rows), rng.integers(0, 300, n_rows),
                     rng.integers(0, 4, n_rows)], 1).astype(np.uint32)
    for top in (0, 60, 120):
        want = oracle.tcrdist_filter(seqs, off, rows, top)
        got = xtn.tcrdist_filter(seqs, off, rows, top)
        assert np.array_equal(_rows(got), want)


@pytest.mark.parametrize("d", [0, 1, 2, 3])
def test_lookup(xtn, d):
    """Groups a lane emits alone, groups spread over warps, one query (split
    between warps) to several a warp, more candidates than the first guess."""
    rng = np.random.default_rng(d)
    refs = (["CASSLGTDTQYF"] * 3000 + ["CASSPGQGAYEQYF"] * 256 + ["CATSDLNEQYF"] * 257
            + ["CA", "", "A" * 25])
    refs += ["".join(rng.choice(list("ACDEFGHIKLMNPQRSTVWY"), rng.integers(0, 26)))
             for _ in range(2000)]
    seqs, off = gen.from_strings([refs[i] for i in rng.permutation(len(refs))])
    idx = xtn.index_build(*_cuda(seqs, off), d)
    for qs in (["CASSLGTDTQYF"], ["A" * 25, "CASSPGQGAYEQYF", "CATSDLNEQYF", ""],
               (refs[2990:3540] + refs[-900:]) * (1 if d == 3 else 7),
               ["CASSLGTDTQYF"] * 300):
        q, qo = gen.from_strings(qs)
        want = oracle.bruteforce_query(seqs, off, q, qo, d, threads=0)
        for _ in range(2):  # the second guess knows the first call's counts
            assert np.array_equal(_rows(xtn.search_query(idx, *_cuda(q, qo), cap=len(want))), want)


@pytest.mark.parametrize("copies,others", [(724, 0), (724, 1400), (725, 0)])
def test_last_step_by_groups(xtn, copies, others):
    """261,726 candidates in groups of 4 sequences, which a block holds, and of
    16, which it does not (the survivors are sorted); one copy more, past the
    limit on candidates."""
    rng = np.random.default_rng(others)
    strs = ["CASSLGTDTQYF"] * copies + [
        "W" + "".join(rng.choice(list("ACDEFGHIKL"), 20)) for _ in range(others)]
    seqs, off = gen.from_strings(strs)
    want = np.stack([*np.triu_indices(copies, 1), np.zeros(copies * (copies - 1) // 2)], 1)
    got = _rows(xtn.search_self(*_cuda(seqs, off), 0, cap=len(want)))
    assert np.array_equal(got, want.astype(np.uint32))
    few = torch.zeros((100, 3), dtype=torch.int32, device="cuda")  # too small a buffer
    n = ctypes.c_int64(0)
    status = xtn.native.lib().xtn_search_self(
        seqs.ctypes.data, off.ctypes.data, len(strs), 0, None, 0, few.data_ptr(), 100,
        ctypes.byref(n), None)
    assert status != 0 and n.value == len(want)
    assert np.array_equal(_rows(few), want[:100].astype(np.uint32))
