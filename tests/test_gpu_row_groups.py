"""The last step by groups where nearly every group has more rows than a block
holds: its warps leave the listing loop at different times, each as a whole."""
import numpy as np
import pytest

import cdr3_synth as gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# empty sequences have one variant, so a pair is one candidate: 1,999,000 of
# them in groups of 8 sequences, up to 16,000 rows each; and 130,816 in groups
# of 2, up to 1,022
@pytest.mark.parametrize("n", [512, 2000])
def test_groups_past_a_blocks_table(n):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2403_09010_gb300 as xtn
    xtn.build()
    seqs, off = gen.from_strings([""] * n)
    do = torch.from_numpy(off).cuda()
    ds = torch.zeros(1, dtype=torch.uint8, device="cuda")
    want = np.stack([*np.triu_indices(n, 1), np.zeros(n * (n - 1) // 2)], 1).astype(np.uint32)
    for _ in range(3):
        got = xtn.search_self(ds, do, 2, cap=len(want))
        assert np.array_equal(got.cpu().numpy().astype(np.uint32), want)
