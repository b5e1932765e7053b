"""Device memory a call takes for its scratch: a search in passes within what
its budget of records stands for, however many passes and spilled partitions."""
import ctypes

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
    torch.zeros(1, device="cuda")
    return pkg


def _cuda(*arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


class PoolPeak:
    """The most bytes of the device's default memory pool in use at a time
    (scratch comes from there) while the block runs, from an empty cache."""
    USED_HIGH = 8  # CU_MEMPOOL_ATTR_USED_MEM_HIGH

    def __init__(self, xtn):
        self.xtn = xtn
        self.cuda = ctypes.CDLL("libcuda.so.1")
        self.pool = ctypes.c_void_p()
        assert self.cuda.cuDeviceGetDefaultMemPool(
            ctypes.byref(self.pool), torch.cuda.current_device()) == 0

    def __enter__(self):
        torch.cuda.synchronize()
        self.xtn.scratch_trim()
        zero = ctypes.c_uint64(0)
        assert self.cuda.cuMemPoolSetAttribute(self.pool, self.USED_HIGH, ctypes.byref(zero)) == 0
        return self

    def __exit__(self, *exc):
        torch.cuda.synchronize()
        high = ctypes.c_uint64(0)
        assert self.cuda.cuMemPoolGetAttribute(self.pool, self.USED_HIGH, ctypes.byref(high)) == 0
        self.bytes = high.value
        return False


def test_passes_take_32_bytes_a_record(xtn):
    """The documented size of a pass, besides the sequences (80 bytes: keys,
    lengths, masks, planes, offsets) and the verified pairs (growing to 1.5
    times their number, and once more where they are sorted)."""
    n, per_pass = 500_000, 20_000_000
    ds, do = _cuda(*gen.generate(n, 5, 0.15, 0.01))
    want = xtn.search_self(ds, do, 2)
    with PoolPeak(xtn) as peak:
        rows, passes = xtn.search_self_streaming(ds, do, 2, max_pass_records=per_pass)
    assert passes >= 3 and torch.equal(rows, want)
    assert peak.bytes <= 32 * per_pass + 80 * n + 8 * (1 << 20) + 3 * 8 * len(want) + (8 << 20)


def test_passes_that_all_spill_take_their_scratch_once(xtn):
    """190 passes of 5,000 records in keys of 300 copies each: every pass has
    partitions that run over (256 regions of about 180 records)."""
    rng = np.random.default_rng(3)
    one = gen.to_strings(*gen.generate(200, 1, 0.0, 0.0))
    strs = [one[k] for k in rng.permutation(np.repeat(np.arange(200), 300))]
    ds, do = _cuda(*gen.from_strings(strs))
    cap = 200 * 300 * 299 // 2 + 2000 * 300 * 300
    want = xtn.search_self(ds, do, 1, cap=cap)
    peaks = []
    for per_pass in (5_000, 20_000):
        with PoolPeak(xtn) as peak:
            xtn.profile_report()
            xtn.profile_enable(True)
            rows, passes = xtn.search_self_streaming(ds, do, 1, max_pass_records=per_pass, cap=cap)
            xtn.profile_enable(False)
            spans = xtn.profile_report()
        assert torch.equal(rows, want)
        peaks.append((peak.bytes, passes, spans["host_scratch_alloc"][0]))
    assert peaks[0][1] > 100 and peaks[0][1] > 3 * peaks[1][1]
    # a pass's buffers, and the few times that the pair words' buffers grow
    assert peaks[0][2] < 80 and peaks[0][0] <= peaks[1][0] + (8 << 20)


class LittleMemory:
    """All of the device's memory but `free` bytes taken, the scratch cache empty."""

    def __init__(self, xtn, free):
        self.xtn, self.free = xtn, free

    def __enter__(self):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.xtn.scratch_trim()
        have = torch.cuda.mem_get_info()[0]
        self.hog = torch.empty(have - self.free, dtype=torch.uint8, device="cuda")

    def __exit__(self, *exc):
        del self.hog
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.xtn.scratch_trim()
        return False


# 104.8 M records (115.5 M in a plan's bound).  With partitions a search takes
# 29 bytes a record and 93 a sequence (3.1 GB), a plan 25 and 28 a pair of its
# capacity (3.2 GB), a build 20 and 10 for the index (3.2 GB); sorted, 17, 17
# and 27 (1.9, 2.3 and 2.9 GB).
@pytest.mark.parametrize("what,free", [("search", 2_500 << 20), ("passes", 2_600 << 20),
                                       ("plan", 2_750 << 20), ("index", 2_870 << 20),
                                       ("search", 8_000 << 20), ("index", 8_000 << 20)])
def test_sorted_where_partitions_do_not_fit(xtn, what, free):
    n, cap = 1_000_000, 400_000
    seqs, off = gen.workload(gen.SELF_1M)
    ds, do = _cuda(seqs, off)
    want = xtn.search_self(ds, do, 2, cap=cap)
    with LittleMemory(xtn, free):
        for _ in range(2):
            xtn.profile_report()
            xtn.profile_enable(True)
            if what == "plan":
                plan = xtn.Plan(off, 2, pair_capacity=6_000_000)
                plan.run(ds)
                got = plan.result(cap=cap, like=ds)
                plan.free()
            elif what == "passes":
                got, _ = xtn.search_self_streaming(ds, do, 2, max_pass_records=120_000_000,
                                                   cap=cap)
            elif what == "index":
                idx = xtn.index_build(ds, do, 2)
                got = want
                info = idx.info()
                idx.free()
                assert info["n_records"] > 104_000_000
            else:
                got = xtn.search_self(ds, do, 2, cap=cap)
            xtn.profile_enable(False)
            kernels = xtn.profile_report()
            assert torch.equal(got, want)
            parted = "k_index_build" if what == "index" else "k_bucket_filter"
            assert (parted in kernels) == (free > 4_000 << 20)
            assert what != "index" or ("k_bucket_sort" in kernels) == (free < 4_000 << 20)
