"""GPU parity of attend_dense_kernel at the edges of its unit counts and cuts, against the fp64 oracle.

bf16 storage, fp32 accumulation: max-abs error <= 1e-2 as in the other attention tests; caches byte for byte."""
import numpy as np
import pytest

import ec_synth as syn
from test_gpu_attend import _check

pytestmark = pytest.mark.gpu


# std_qk 4: scores of standard deviation 16, which send a unit through its second pass
@pytest.mark.parametrize("std_qk", [None, 4.0])
@pytest.mark.parametrize("Hq,Hkv,L,n,cut", [
    (9, 9, 300, 300, "cut_units=0x1"),       # 18 units, one above the one-tile kernel's; three tiles, the last ragged
    (32, 8, 256, 256, "cut_units=0x1"),      # 32 units of one pair of row tiles, two key tiles
    (17, 17, 257, 257, "cut_units=0x1"),     # a row tile of one row
    (4, 4, 2048, 2048, "cut_units=32x4"),    # nothing but cut units: 4 parts
    (7, 7, 1500, 1500, "cut_units=42x3"),    # 3 parts: a merge share that is no whole number of fours
    (2, 2, 2560, 2560, "cut_units=20x5"),    # 5 parts
    (2, 2, 2600, 2304, "cut_units=18x5"),    # 5 parts of 21 tiles, fewer rows than keys (an index list)
])
def test_recompute_steps_with_few_units_and_any_number_of_parts(Hq, Hkv, L, n, cut, std_qk):
    import paper_2603_18489_b200 as ec

    w = syn.Workload(97, f"h{Hq}_l{L}", syn.BF16, 1, Hq, Hkv, 128, L - 64, 64, 32, 2, 1024)
    full = n == L
    got = ec.ec_attend_kernel_name(ec.make_desc(1, L, Hq, Hkv, 128, syn.BF16), n, True, not full)
    assert "attend_dense_kernel" in got and cut in got, got
    idx = None if full else syn.arbitrary_active_idx(1, L, n, seed=6)
    t = syn.attn_inputs(w, n, active_idx=idx, std_qk=std_qk, salt=5)
    rng = np.random.Generator(np.random.PCG64(L + Hq))
    rows = sorted(set(rng.choice(n, min(n, 16), replace=False).tolist() + [0, n - 1]))
    _check(w, t, row_sel=rows)
