"""Which kernel ec_attend picks for each benchmark shape (host-only query, no launch).  The parity tests in
test_gpu_attend.py / test_gpu_config5.py run these very shapes against the oracle; this table pins the kernel
behind each of them, so a change of the dispatch cannot leave a kernel without a parity test unnoticed.
The plans assume 148 SMs (the B200's count, also the library's default when no device can be queried); cluster sizes
are not pinned here, because with a device present the library asks the runtime how many clusters stay resident."""
import pytest

import ec_synth as syn

# (workload, batch override, active rows) -> kernel family with its instantiation, on the skip step
SKIP_STEP = [
    ("c2_llada_l768", None, 34, "attend_skip_keys_kernel<48>"),
    ("c3_dream_l768", None, 34, "attend_skip_keys_kernel<48>"),
    ("c4_llada_l2048", None, 33, "attend_skip_keys_kernel<48>"),
    ("c4_llada_l2048", None, 40, "attend_skip_keys_kernel<48>"),
    ("c5_llada_l4096", None, 34, "attend_skip_keys_kernel<48>"),
    ("c5_llada_l4096", 2, 34, "attend_skip_keys_kernel<48>"),
    ("c5_llada_l4096_b8", None, 34, "attend_skip_kernel<1>"),       # beyond one wave of one-CTA-per-SM clusters
    ("c5_llada_l4096", 5, 34, "attend_skip_kernel<1>"),
    ("c4_dream_l2048", None, 34, "attend_skip_keys_kernel<48>"),
    ("c5_dream_l4096", None, 34, "attend_skip_keys_kernel<48>"),
    ("c5_llada_l4096", None, 96, "attend_skip_keys_kernel<96>"),    # the paper's default budget k = 64
    ("c5_llada_l4096_b8", None, 96, "attend_skip_kernel<1>"),
    ("c5_dream_l4096", None, 96, "attend_skip_keys_kernel<96>"),
    ("c1_tiny_fp32", None, 34, "refresh_kernel + attend_f32_kernel"),
]

RECOMPUTE_STEP = [
    ("c1_tiny_fp32", None, "refresh_kernel + attend_f32_kernel"),
    ("c2_llada_l768", None, "attend_dense_kernel"),
    ("c3_dream_l768", None, "attend_dense_kernel"),
    ("c4_llada_l2048", None, "attend_dense_kernel"),
    ("c5_llada_l4096", None, "attend_dense_kernel"),
    ("c5_llada_l4096_b8", None, "attend_dense_kernel"),
    ("c4_dream_l2048", None, "attend_dense_kernel"),
    ("c5_dream_l4096", None, "attend_dense_kernel"),
]


def _desc(name, batch):
    import paper_2603_18489_b200 as ec

    w = syn.WORKLOADS[name]
    return ec, ec.make_desc(batch or w.batch, w.ctx_len, w.n_q_heads, w.n_kv_heads, w.head_dim, w.dtype), w


@pytest.mark.parametrize("name,batch,n,kernel", SKIP_STEP)
def test_kernel_of_each_benchmark_skip_step(name, batch, n, kernel):
    ec, d, w = _desc(name, batch)
    got = ec.ec_attend_kernel_name(d, n, True, True)
    assert got.startswith(kernel), got
    if "grid=" in got:      # the cluster splits the key tiles; the grid's second dimension covers every (sequence, head)
        gx, gy = (int(v) for v in got.split("grid=(")[1].split(")")[0].split(","))
        assert gy % ((batch or w.batch) * w.n_kv_heads) == 0 and f"cluster={gx}" in got


@pytest.mark.parametrize("name,batch,kernel", RECOMPUTE_STEP)
def test_kernel_of_each_benchmark_recompute_step(name, batch, kernel):
    ec, d, w = _desc(name, batch)
    got = ec.ec_attend_kernel_name(d, w.ctx_len, True, False)
    assert got.startswith(kernel), got


def test_other_instantiations_and_fallbacks_are_reachable():
    """Every kernel (and template instantiation) of the attention path, with a shape that reaches it; each of
    these shapes has a parity case in test_gpu_attend.py."""
    import paper_2603_18489_b200 as ec

    def name(B, L, Hq, Hkv, D, dtype, n, idx=True):
        return ec.ec_attend_kernel_name(ec.make_desc(B, L, Hq, Hkv, D, dtype), n, True, idx)

    assert name(2, 1000, 8, 8, 128, syn.BF16, 56).startswith("attend_skip_keys_kernel<64>")
    assert name(2, 333, 6, 3, 128, syn.BF16, 100).startswith("attend_skip_keys_kernel<64>")  # 200 packed rows
    assert name(1, 640, 4, 4, 128, syn.BF16, 256).startswith("attend_skip_keys_kernel<96>")  # three row chunks
    assert "fresh_tiles=1" in name(1, 768, 32, 32, 128, syn.BF16, 34)      # the refreshed rows are attended as one extra tile
    assert "fresh_tiles=2" in name(1, 4096, 32, 32, 128, syn.BF16, 160)
    assert "fresh_tiles=0" in ec.ec_attend_kernel_name(ec.make_desc(1, 768, 32, 32, 128, syn.BF16), 34, False, True)
    assert name(2, 768, 32, 32, 128, syn.BF16, 128).startswith("attend_skip_kernel<1> grid=(4,64) cluster=4")
    assert name(3, 768, 32, 32, 128, syn.BF16, 128).startswith("attend_skip_kernel<1> grid=(3,96) cluster=3")
    assert name(2, 768, 32, 32, 128, syn.BF16, 160).startswith("attend_skip_kernel<2> grid=(2,64) cluster=2")
    assert name(8, 4096, 32, 32, 128, syn.BF16, 200).startswith("attend_skip_kernel<2> grid=(1,256) cluster=1")
    assert name(2, 65, 6, 3, 128, syn.BF16, 65, idx=False).startswith("attend_skip_keys_kernel<96>")
    assert name(2, 259, 4, 2, 128, syn.BF16, 259, idx=False) == "refresh_kernel + attend_tc_kernel"
    assert name(2, 130, 6, 3, 64, syn.BF16, 17) == "refresh_kernel + attend_mma_kernel"
    assert name(2, 130, 6, 3, 64, syn.F32, 17) == "refresh_kernel + attend_f32_kernel"
    # the dense kernel cuts the units of its last, partial wave along the keys when that pays (148 SMs assumed)
    assert "whole_units=444 cut_units=68x2" in name(1, 4096, 32, 32, 128, syn.BF16, 4096, idx=False)
    assert "whole_units=444 cut_units=4x8" in name(1, 4096, 28, 4, 128, syn.BF16, 4096, idx=False)
    assert "cut_units=0x1" in name(1, 2048, 32, 32, 128, syn.BF16, 2048, idx=False)
    assert "cut_units=0x1" in name(8, 4096, 32, 32, 128, syn.BF16, 4096, idx=False)
    assert ec.ec_attend_kernel_name(ec.make_desc(1, 64, 4, 4, 64, syn.F32), 65, True, True) == ""   # rejected


@pytest.mark.parametrize("Hq,Hkv", [(32, 32), (28, 4), (9, 9)])
def test_every_part_of_a_cut_unit_holds_key_tiles(Hq, Hkv):
    """The last wave of a recompute step is cut along the keys: whatever the number of key tiles, its parts are level
    and none of them is empty (a part without a tile would wait for data that nobody loads)."""
    import re

    import paper_2603_18489_b200 as ec

    n_cut = 0
    for B in range(1, 9):
        for tiles in range(1, 65):
            for L, n in ((128 * tiles, 128 * tiles), (128 * tiles - 57, 128 * tiles - 57), (128 * tiles, min(300, 128 * tiles))):
                got = ec.ec_attend_kernel_name(ec.make_desc(B, L, Hq, Hkv, 128, syn.BF16), n, True, n != L)
                if not got.startswith(("attend_dense", "refresh_kernel + attend_dense")):
                    continue
                cut, parts, lo, hi = (int(v) for v in re.search(r"cut_units=(\d+)x(\d+) part_tiles=(-?\d+)\.\.(\d+)", got).groups())
                assert lo == tiles // parts and hi == -(-tiles // parts), got
                assert lo >= 4 or parts == 1, got
                n_cut += cut > 0
    assert n_cut > 50


@pytest.mark.parametrize("B,L,Hq,Hkv,n,fresh,kernel", [
    # 64-wide heads: mma.sync takes the time behind the colon, the dense kernel the other
    (1, 1000, 9, 9, 257, True, "attend_mma_kernel"),     # 9.2 us: 14.8
    (1, 449, 9, 9, 257, True, "attend_mma_kernel"),      # 7.4: 11.0
    (2, 700, 9, 9, 129, True, "attend_mma_kernel"),      # 9.9: 13.5
    (1, 700, 17, 17, 160, True, "attend_mma_kernel"),    # 11.0: 13.6
    (4, 700, 6, 2, 129, True, "attend_mma_kernel"),      # 10.9: 13.6
    (4, 300, 24, 8, 257, False, "attend_mma_kernel"),    # 10.6: 15.0
    (32, 129, 24, 8, 129, True, "attend_mma_kernel"),    # a recompute step, 32.0: 42.1
    (1, 129, 17, 17, 17, False, "attend_mma_kernel"),    # 3.6: 4.7
    (16, 1024, 32, 8, 48, True, "attend_mma_kernel"),    # 35.0: 46.7
    (1, 300, 9, 9, 300, True, "attend_dense_kernel<64>"),     # a recompute step, 9.0: 7.8
    (4, 1000, 24, 8, 96, True, "attend_dense_kernel<64>"),    # 23.9: 13.6
    (8, 1024, 9, 9, 128, True, "attend_dense_kernel<64>"),    # 30.2: 14.5
    (1, 1500, 12, 12, 384, True, "attend_dense_kernel<64>"),  # 23.0: 15.8
    (32, 449, 32, 4, 257, True, "attend_dense_kernel<64>"),   # more than 256 rows, more units than SMs
])
def test_64_wide_heads_run_on_the_faster_kernel(B, L, Hq, Hkv, n, fresh, kernel):
    import paper_2603_18489_b200 as ec

    got = ec.ec_attend_kernel_name(ec.make_desc(B, L, Hq, Hkv, 64, syn.BF16), n, fresh, n != L)
    assert got.split(" grid")[0].split(" + ")[-1] == kernel, got
