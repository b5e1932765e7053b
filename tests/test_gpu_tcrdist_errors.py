"""The TCRdist filter leaves the caller's rows alone when it refuses the
sequences, with either number of rows a thread."""
import ctypes

import pytest

import cdr3_synth as gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("entry", ["xtn_tcrdist_filter", "xtn_tcrdist_filter_noalloc"])
@pytest.mark.parametrize("n_rows", [3, 262_145])
@pytest.mark.parametrize("bad,status", [("CAXSF", "XTN_ERR_BAD_RESIDUE"),
                                        ("A" * 26, "XTN_ERR_SEQ_TOO_LONG")])
def test_out_is_left_alone(entry, n_rows, bad, status):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2403_09010_gb300 as xtn
    xtn.build()
    seqs, off = gen.from_strings(["CASSF", "CASF", bad])
    ds, do = torch.from_numpy(seqs).cuda(), torch.from_numpy(off).cuda()
    rows = torch.tensor([[0, 1, 1]], dtype=torch.int32, device="cuda").repeat(n_rows, 1)
    out = torch.full((n_rows, 3), 77, dtype=torch.int32, device="cuda")
    n_out = ctypes.c_int64(5)

    def call(n_seqs):
        return getattr(xtn.native.lib(), entry)(
            ds.data_ptr(), do.data_ptr(), n_seqs, rows.data_ptr(), n_rows, 100, out.data_ptr(),
            ctypes.byref(n_out), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))

    assert call(3) == getattr(xtn.native, status) and n_out.value == 0
    assert bool((out == 77).all())
    assert call(2) == 0 and n_out.value == n_rows  # the first two by themselves
    assert torch.equal(out, rows)
