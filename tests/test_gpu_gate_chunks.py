"""GPU parity of the gate where rows are cut into s or s + 1 chunks, against the fp64 oracle (tolerances of test_gpu_gate)."""
import numpy as np
import pytest
import torch

import ec_synth as syn
import oracle
from _util import to_dev
from test_gpu_gate import ENT_TOL, _compare, _run_gpu
from test_gpu_gate_decode import _check as _check_decode, _logits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [syn.F32, syn.BF16])
@pytest.mark.parametrize("R,rps,V,stride", [
    (256, 32, 9001, 9008),    # 2 or 3 chunks (bf16), the change inside a sequence; ragged vocabulary, padded rows
    (592, 16, 4100, 4104),    # as many rows as places: one chunk a row
    (576, 64, 4100, 4104),    # 16 places to spare: one chunk a row
    (350, 35, 4100, 4104),    # one chunk or two (bf16)
    (296, 8, 6600, 6600),     # two or three, and no row has three (bf16)
    (593, 593, 2100, 2104),   # more rows than places: equal chunks
    (42, 7, 40001, 40008),    # 14 or 15
    (130, 65, 20001, 20008),  # 4 or 5 (bf16), two ticket levels
    (19, 19, 126464, 126464), # 31 or 32: the most that one CTA finishes; the 32nd is empty
    (18, 6, 126464, 126464),  # 32 or 33 would be one too many: equal chunks
    (10, 5, 152064, 152064),  # 59 or 60 (38 equal ones would be too many as well), two ticket levels
    (3, 3, 400002, 400008),   # the limit of splits
    (32, 32, 36863, 36864),   # equal chunks
    (32, 32, 38911, 38912),   # one column short of the smallest chunk: equal chunks
    (32, 32, 38912, 38912),   # the smallest chunk
])
def test_rows_cut_into_unequal_numbers_of_chunks(dtype, R, rps, V, stride):
    d = syn.logits_rows(R, V, dtype, cfg_id=60 + R % 7, row_stride=stride)
    flags = syn.decoded_flags(R, max(1, rps // 2), rps, cfg_id=61)
    o = oracle.entropy_gate(d["logits"], dtype, V, flags, 2.0, rps)
    for _ in range(2):   # (the tickets are zero again)
        _compare(_run_gpu(d["logits"], dtype, V, flags, 2.0, rps), o, 2.0)


@pytest.mark.parametrize("dtype,R,rps,V,stride", [
    (syn.BF16, 256, 32, 9001, 9008),    # 2 or 3 chunks, the change in the middle of the sixth sequence
    (syn.F32, 42, 7, 40001, 40008),     # 14 or 15, in the sixth
    (syn.BF16, 350, 35, 4100, 4104),    # 1 or 2, in the fourth
    (syn.F32, 20, 4, 126464, 126464),   # 29 or 30, in the second
])
def test_decoding_and_metrics_where_a_sequence_has_rows_of_both_kinds(dtype, R, rps, V, stride):
    """One CTA finishes a sequence; it counts the partials of rows with s and with s + 1 chunks."""
    import paper_2603_18489_b200 as ec

    lg = _logits(R, V, dtype, 62, n_spiked=R // 3, stride=stride)
    masked = (np.random.Generator(np.random.PCG64(R)).random(R) < 0.7).astype(np.uint8)
    for _ in range(2):
        _check_decode(lg, dtype, V, masked, 0.9, 1.5, rps)
    flags = syn.decoded_flags(R, max(1, rps // 2), rps, cfg_id=63)
    o = oracle.entropy_gate(lg, dtype, V, flags, 1.5, rps)
    m = oracle.gate_metrics(o["entropy"], o["conf"], flags, rps)
    g = ec.ec_entropy_gate_metrics(to_dev(lg), V, rps, to_dev(flags), 1.5)
    g = {k: v.cpu().numpy() for k, v in g.items()}
    _compare(g, o, 1.5)
    n_dec = flags.reshape(-1, rps).sum(axis=1)
    assert np.all(np.abs(g["entropy_sum"].astype(np.float64) - m["entropy_sum"]) <= ENT_TOL * n_dec)
    assert np.all(np.abs(g["max_conf"].astype(np.float64) - m["max_conf"]) <= 1e-5 * m["max_conf"])


def _chunks_of_a_call(R, rps, V, dtype):
    """Rows and the number of partials that a call leaves in its workspace, behind the tickets and one word a row."""
    import paper_2603_18489_b200 as ec

    ws = ec.new_workspace(ec.ec_entropy_gate_workspace_bytes(R, V))
    flags = torch.ones(R, dtype=torch.uint8, device="cuda")
    ec.ec_entropy_gate(torch.randn(R, V, device="cuda").to(dtype), V, rps, flags, 1.5, workspace=ws)
    return int(ws[(R * 12 + 15) // 16 * 16:].view(-1, 16).any(1).sum())


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("R,rps", [(10, 10), (12, 4), (16, 16), (18, 6), (19, 19)])
def test_rows_that_one_cta_can_finish_are_not_cut_for_two_levels(dtype, R, rps):
    """A row of 33 chunks and more is finished by two levels of tickets, 1 us later (5.3 -> 6.5 at 16 rows); equal chunks of
    whole slabs are 31 of these rows."""
    assert _chunks_of_a_call(R, rps, 126464, dtype) <= 32 * R


@pytest.mark.parametrize("R,rps,V,dtype,chunks", [
    (148, 37, 32000, torch.bfloat16, 4 * 148),     # as many places as equal chunks
    (280, 28, 64000, torch.bfloat16, 2 * 280),     # 32 rows could have a third chunk
    (296, 37, 32000, torch.bfloat16, 2 * 296),
    (425, 25, 32000, torch.bfloat16, 425),         # whole rows would be the longest chunks anyway
    (592, 37, 4104, torch.bfloat16, 592),
    (80, 8, 100352, torch.float32, 7 * 80),        # large chunks in fp32
    (400, 40, 32000, torch.bfloat16, 400), (400, 40, 126464, torch.bfloat16, 592),
    (256, 32, 126464, torch.bfloat16, 592), (72, 36, 32000, torch.float32, 592),
])
def test_rows_are_cut_unequally_only_where_that_is_faster(R, rps, V, dtype, chunks):
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the counts are those of 148 SMs")
    assert _chunks_of_a_call(R, rps, V, dtype) == chunks
