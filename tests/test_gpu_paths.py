"""GPU parity at the sizes where single paths of the kernels can go wrong: cluster sizes whose CTAs merge unequal
shares of the output, references of the softmax taken from the rare path, edges of tiles and of dispatch rules.
Each against the fp64 oracle, with the tolerances of test_gpu_attend.py."""
import numpy as np
import pytest

import ec_synth as syn
from test_gpu_attend import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n", [(64, 1), (257, 34), (500, 33), (640, 48), (769, 34), (900, 60), (896, 96)])
def test_cluster_sizes_with_unequal_output_shares(L, n):
    """Two heads, so the keys split over as many CTAs as there are tiles (one to eight with the fresh rows' own CTA):
    the CTAs own 128, 64, 48, 32, 24 or 16 output columns, the last ones fewer or none."""
    w = syn.Workload(97, "clusters", syn.BF16, 1, 2, 2, 128, 0, L, 1, 0, 64)
    t = syn.attn_inputs(w, n, active_idx=syn.arbitrary_active_idx(1, L, n, seed=17 * L + n), std_qk=0.9, std_v=0.5)
    _check(w, t)
    _check(w, t, refresh=False)


@pytest.mark.parametrize("std,L", [(0.3, 1024), (2.5, 1024), (14.0, 600)])
def test_first_keys_of_a_tile_all_refreshed(std, L):
    """The first 32 keys of every second tile are refreshed, so no cached key of the warp that supplies a CTA's first
    reference counts and the reference comes from the rare path; with std 14 scores exceed references by far."""
    idx = np.concatenate([np.arange(i, i + 32) for i in range(0, min(L, 700), 256)])[None].astype(np.int32)
    w = syn.Workload(98, "stale", syn.BF16, 1, 8, 8, 128, 0, L, 1, 0, 64)
    _check(w, syn.attn_inputs(w, idx.shape[1], active_idx=idx, std_qk=std, std_v=0.5))


@pytest.mark.parametrize("B,Hq,Hkv,L,n", [(5, 32, 32, 130, 1), (5, 32, 32, 300, 48), (20, 16, 8, 257, 20), (19, 8, 8, 128, 49),
                                          (5, 32, 32, 700, 64), (5, 32, 32, 64, 33)])
def test_many_heads_with_few_rows(B, Hq, Hkv, L, n):
    """More kv heads than SMs, one CTA each with the keys on the M axis: 48 and 64 query slots, grouped queries, ragged
    tiles, a context of a single tile that is half refreshed; with and without fresh rows, flat and peaky scores."""
    import paper_2603_18489_b200 as ec

    w = syn.Workload(99, "many_heads", syn.BF16, B, Hq, Hkv, 128, 0, L, 1, 0, 64)
    assert "keys_on_m" in ec.ec_attend_kernel_name(ec.make_desc(B, L, Hq, Hkv, 128, syn.BF16), n, True, True)
    idx = syn.arbitrary_active_idx(B, L, n, seed=19 * L + n)
    for std in (0.5, 6.0):
        t = syn.attn_inputs(w, n, active_idx=idx, std_qk=std, std_v=0.5)
        _check(w, t)
        _check(w, t, refresh=False)


@pytest.mark.parametrize("Hq,Hkv,L,cut", [(10, 5, 1100, "whole_units=0 cut_units=50x2"), (33, 33, 1100, "whole_units=148 cut_units=17x2"),
                                          (5, 5, 2500, "whole_units=0 cut_units=50x2")])
def test_cut_units_alone_and_with_a_single_row_tile(Hq, Hkv, L, cut):
    """Recompute steps with no whole unit beside the cut ones, and with units of one row tile among the cut ones;
    moderate scores, and peaky ones for which some parts of a unit run their second pass and others do not."""
    import paper_2603_18489_b200 as ec

    w = syn.Workload(100, "cut", syn.BF16, 1, Hq, Hkv, 128, 0, L, 1, 0, 64)
    assert cut in ec.ec_attend_kernel_name(ec.make_desc(1, L, Hq, Hkv, 128, syn.BF16), L, True, False)
    rows = sorted(set(np.random.Generator(np.random.PCG64(L)).choice(L, 40, replace=False).tolist() + [0, L - 1]))
    for std in (0.5, 8.0):
        _check(w, syn.attn_inputs(w, L, std_qk=std, std_v=0.5, salt=Hq), row_sel=rows)


@pytest.mark.parametrize("H,L,cut", [(9, 4100, "cut_units=5x8 part_tiles=4..5"), (9, 4400, "cut_units=14x8 part_tiles=4..5"),
                                     (6, 6200, "cut_units=2x8 part_tiles=6..7"), (17, 2200, "cut_units=5x4 part_tiles=4..5")])
def test_cut_units_of_uneven_parts(H, L, cut):
    """Key tiles that the number of parts does not divide: the cut units are the last ones, those of the last heads."""
    import paper_2603_18489_b200 as ec

    w = syn.Workload(104, "uneven", syn.BF16, 1, H, H, 128, 0, L, 1, 0, 64)
    assert cut in ec.ec_attend_kernel_name(ec.make_desc(1, L, H, H, 128, syn.BF16), L, True, False)
    rows = sorted(set(np.random.Generator(np.random.PCG64(L)).choice(L, 40, replace=False).tolist() + [0, L - 1]))
    for std in (0.5, 8.0):
        _check(w, syn.attn_inputs(w, L, std_qk=std, std_v=0.5, salt=H), row_sel=rows)


@pytest.mark.parametrize("dtype", [syn.BF16, syn.F32])
@pytest.mark.parametrize("V", [8, 2048, 2056, 4096, 2048 * 3 + 40, 2048 * 6, 2048 * 7 + 1003])
def test_first_maximum_among_the_vectors_of_a_thread(dtype, V):
    """Rows cut into one chunk, one to eight vectors a thread: the maximum planted in every vector of a pair in turn,
    with copies of it in the next vector of the same thread, in the last columns and beside it."""
    import oracle
    from test_gpu_gate import _compare, _run_gpu

    R, V0 = 608, V // 8 * 8
    x = np.random.Generator(np.random.PCG64(V)).normal(0, 2, (R, V0 + 16)).astype(np.float32)
    for r in range(R):
        at = (r * 1031 + r // 8 * 7) % V
        x[r, [c for c in (at, at + 1, at + 2048, at + 4096, V - 1) if c < V]] = 9.0 + r % 5
    st = syn.encode(x, dtype)
    flags = np.ones(R, np.uint8)
    _compare(_run_gpu(st, dtype, V, flags, 2.0, 32), oracle.entropy_gate(st, dtype, V, flags, 2.0, 32), 2.0)


@pytest.mark.parametrize("B,Hq,Hkv,L,n", [(1, 4, 2, 200, 33), (2, 6, 2, 900, 44), (1, 3, 1, 130, 48), (8, 8, 8, 300, 65), (1, 12, 4, 64, 64)])
def test_row_tiles_of_48_rows(B, Hq, Hkv, L, n):
    """64-wide heads, two to four row tiles of at most 48 rows on mma.sync: remainders in the last tile, ragged key tiles, one
    key tile and several; with and without fresh rows.  (8 x 300 with 65 rows runs on the dense kernel.)"""
    w = syn.Workload(101, "d64_tiles", syn.BF16, B, Hq, Hkv, 64, 0, L, 1, 0, 64)
    t = syn.attn_inputs(w, n, active_idx=syn.arbitrary_active_idx(B, L, n, seed=L + n), std_qk=0.9, std_v=0.5)
    _check(w, t)
    _check(w, t, refresh=False)


@pytest.mark.parametrize("B,Hq,Hkv,L", [(2, 4, 2, 1), (1, 2, 2, 64), (3, 6, 2, 65), (1, 4, 1, 200), (2, 8, 8, 449)])
def test_recompute_steps_of_64_wide_heads(B, Hq, Hkv, L):
    """K/V tiles by TMA out of the token-major fresh rows and out of the cache: one key, whole and ragged tiles.  (3 x 65 and
    2 x 449 run on the dense kernel, the others on mma.sync.)"""
    w = syn.Workload(102, "d64_full", syn.BF16, B, Hq, Hkv, 64, 0, L, 1, 0, 64)
    t = syn.attn_inputs(w, L, std_qk=0.9, std_v=0.5)
    _check(w, t)
    _check(w, t, refresh=False)


@pytest.mark.parametrize("B,Hq,Hkv,L,n", [(64, 12, 4, 500, 40),    # one CTA walks all eight key tiles
                                          (32, 12, 4, 500, 30),    # the same with row tiles of 48 rows
                                          (16, 12, 4, 700, 48),    # three of 48, two CTAs of six and five tiles
                                          (1, 1, 1, 2048, 2048),   # a recompute step: eight CTAs of four tiles
                                          (1, 2, 2, 2000, 2000)])  # six CTAs, the last with two tiles, one of them ragged
def test_mma_sync_kernel_refills_its_stages(B, Hq, Hkv, L, n):
    """64-wide heads on mma.sync, four and more key tiles a CTA on three stages: an index list with fresh rows, the cache by
    TMA without them, the fresh rows by TMA on a recompute step."""
    import paper_2603_18489_b200 as ec

    for fresh in (True, False):
        got = ec.ec_attend_kernel_name(ec.make_desc(B, L, Hq, Hkv, 64, syn.BF16), n, fresh, n != L)
        assert got.endswith("attend_mma_kernel"), got
    w = syn.Workload(105, "d64_ring", syn.BF16, B, Hq, Hkv, 64, 0, L, 1, 0, 64)
    idx = None if n == L else syn.arbitrary_active_idx(B, L, n, seed=L + n)
    rows = None if n < L else sorted(set(np.random.Generator(np.random.PCG64(L)).choice(n, 40, replace=False).tolist() + [0, n - 1]))
    t = syn.attn_inputs(w, n, active_idx=idx, std_qk=0.9, std_v=0.5)
    _check(w, t, row_sel=rows)
    _check(w, t, row_sel=rows, refresh=False)


@pytest.mark.parametrize("B,Hq,Hkv,D,L,n", [(1, 2, 1, 64, 70, 35), (1, 4, 4, 64, 256, 2), (1, 4, 4, 64, 256, 34), (1, 3, 1, 128, 33, 17),
                                            (1, 8, 8, 128, 300, 40), (2, 6, 2, 64, 161, 48), (6, 8, 8, 64, 300, 40)])
def test_fp32_row_tiles_of_8_16_and_32_rows(B, Hq, Hkv, D, L, n):
    """Row tiles of every height, remainders in the last one, keys split over three to eight CTAs and uneven shares."""
    w = syn.Workload(103, "f32_tiles", syn.F32, B, Hq, Hkv, D, 0, L, 1, 0, 64)
    t = syn.attn_inputs(w, n, active_idx=syn.arbitrary_active_idx(B, L, n, seed=L + n), std_qk=0.9, std_v=0.5)
    _check(w, t)
    _check(w, t, refresh=False)
