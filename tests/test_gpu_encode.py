"""Encoding and distances at the edges of a warp's span: letters that start on
every byte of a word, sequence counts around a warp and a block, empty and
longest sequences, every radius, against the CPU oracle."""
import numpy as np
import pytest

import cdr3_synth as gen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 31, 33, 257])
def test_letters_on_any_byte(shift, n):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2403_09010_gb300 as xtn
    xtn.build()
    rng = np.random.default_rng(10 * n + shift)
    L = rng.choice([0, 1, 2, 3, 8, 24, 25], n)
    base = ["".join(rng.choice(list("ACY"), l)) for l in L]
    seqs, off = gen.from_strings(base)
    raw = torch.zeros(seqs.size + 8, dtype=torch.uint8, device="cuda")
    raw[shift:shift + seqs.size] = torch.from_numpy(seqs).cuda()
    ds = raw[shift:shift + seqs.size]
    do = torch.from_numpy(off).cuda()
    for d in range(4):
        want = oracle.bruteforce_self(seqs, off, d)
        got = xtn.search_self(ds, do, d, cap=n * n + 1).cpu().numpy().astype(np.uint32)
        assert np.array_equal(got, want)
    want = oracle.bruteforce_self(seqs, off, 2, "hamming")
    got = xtn.search_self(ds, do, 2, cap=n * n + 1, metric="hamming").cpu().numpy()
    assert np.array_equal(got.astype(np.uint32), want)
