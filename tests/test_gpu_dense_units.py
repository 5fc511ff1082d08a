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


@pytest.mark.parametrize("std_qk", [None, 4.0])
@pytest.mark.parametrize("B,Hq,Hkv,L,n,cut", [
    (1, 17, 17, 129, 129, "whole_units=17"),     # one key of a second tile, one row of a second row tile
    (2, 12, 4, 300, 300, "whole_units=48"),      # grouped query heads, a ragged third tile
    (1, 7, 7, 1500, 1500, "cut_units=42x3"),
    (1, 2, 2, 2560, 2560, "cut_units=20x5"),
    (2, 40, 8, 260, 259, "whole_units=160"),     # an index list, two rounds of units
    (4, 24, 8, 500, 96, "whole_units=96"),       # a partial step
])
def test_heads_of_64_on_the_dense_kernel(B, Hq, Hkv, L, n, cut, std_qk):
    import paper_2603_18489_b200 as ec

    w = syn.Workload(98, f"d64_h{Hq}_l{L}", syn.BF16, B, Hq, Hkv, 64, L - 64, 64, 32, 2, 1024)
    full = n == L
    got = ec.ec_attend_kernel_name(ec.make_desc(B, L, Hq, Hkv, 64, syn.BF16), n, True, not full)
    assert "attend_dense_kernel<64>" in got and cut in got, got
    idx = None if full else syn.arbitrary_active_idx(B, L, n, seed=7)
    t = syn.attn_inputs(w, n, active_idx=idx, std_qk=std_qk, salt=6)
    rng = np.random.Generator(np.random.PCG64(L + Hq))
    rows = sorted(set(rng.choice(n, min(n, 16), replace=False).tolist() + [0, n - 1]))
    _check(w, t, row_sel=rows)


def test_small_and_packed_steps_of_64_wide_heads_stay_on_mma_sync():
    import paper_2603_18489_b200 as ec

    for B, L, Hq, Hkv, n, idx in [(1, 449, 8, 8, 449, False), (4, 1000, 12, 4, 48, True), (64, 500, 12, 4, 40, True),
                                  (8, 1000, 24, 8, 34, True), (1, 1000, 24, 24, 96, True)]:
        got = ec.ec_attend_kernel_name(ec.make_desc(B, L, Hq, Hkv, 64, syn.BF16), n, True, idx)
        assert got == "refresh_kernel + attend_mma_kernel", (B, L, Hq, Hkv, n, got)


@pytest.mark.parametrize("B,Hq,Hkv,L,D,layers", [(2, 28, 4, 1531, 128, 4), (4, 32, 32, 1024, 128, 3), (1, 32, 32, 3000, 128, 3),
                                                 (4, 24, 8, 1000, 64, 4)])
def test_passes_without_synchronisation_repeat_their_outputs(B, Hq, Hkv, L, D, layers):
    """Layers back to back, several waves of units each: the kernel adds in a fixed order, so every pass gives the same bits.
    (Ring slots that were refilled under a product showed here and in no single call.)  The first pass is compared with
    float32 products of the same bf16 inputs: 2e-2 of the largest output, which a key tile in another's place exceeds."""
    import torch

    import paper_2603_18489_b200 as ec

    g = torch.Generator(device="cuda")
    g.manual_seed(L)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.bfloat16)

    d = ec.make_desc(B, L, Hq, Hkv, D, torch.bfloat16)
    st = [(normal(B, L, Hq, D), normal(B, L, Hkv, D), normal(B, L, Hkv, D), normal(B, Hkv, L, D), normal(B, Hkv, L, D),
           torch.empty(B, L, Hq, D, device="cuda", dtype=torch.bfloat16)) for _ in range(layers)]
    assert "attend_dense_kernel" in ec.ec_attend_kernel_name(d, L, True, False)

    def one_pass():
        for q, kn, vn, kc, vc, out in st:
            ec.ec_attend(d, q, kn, vn, kc, vc, None, out=out)

    one_pass()
    torch.cuda.synchronize()
    first = [s[-1].clone() for s in st]
    for q, kn, vn, kc, vc, out in st:
        assert torch.equal(kc, kn.transpose(1, 2)) and torch.equal(vc, vn.transpose(1, 2))
        for b in range(B):
            for h in range(0, Hq, 5):
                k, v = kn[b, :, h * Hkv // Hq].float(), vn[b, :, h * Hkv // Hq].float()
                ref = torch.softmax(q[b, :, h].float() @ k.T / D ** 0.5, -1) @ v
                assert (out[b, :, h].float() - ref).abs().max() <= 2e-2 * ref.abs().max(), (b, h)
    for _ in range(12):
        for _ in range(3):
            one_pass()
        torch.cuda.synchronize()
        for s, f in zip(st, first):
            assert torch.equal(s[-1], f)


def test_cut_units_run_at_once():
    """The clusters of a cut last wave are no more than the device keeps resident, or the last of them make a second round: 48
    units of 12 to 16 tiles, which three parts each would fit by the number of SMs alone, and every count of units around."""
    import re

    import paper_2603_18489_b200 as ec

    seen = set()
    for D, n in ((128, 300), (64, 200)):
        for L in range(1024, 4097, 256):
            for units in range(17, 148):
                heads = units // 2 if D == 128 else units
                got = ec.ec_attend_kernel_name(ec.make_desc(1, L, heads, heads, D, syn.BF16), n, True, True)
                m = re.search(r"cut_units=(\d+)x(\d+) part_tiles=\d+\.\.\d+( at_once=(\d+))?$", got)
                if m and int(m[1]):
                    assert m[3] and int(m[1]) <= int(m[4]), got
                    seen.add(int(m[2]))
    assert seen >= {2, 3, 4, 5, 6}
