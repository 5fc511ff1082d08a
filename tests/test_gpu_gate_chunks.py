"""GPU parity of the gate where rows are cut into s or s + 1 chunks, against the fp64 oracle (tolerances of test_gpu_gate)."""
import pytest

import ec_synth as syn
import oracle
from test_gpu_gate import _compare, _run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [syn.F32, syn.BF16])
@pytest.mark.parametrize("R,rps,V,stride", [
    (256, 32, 9001, 9008),    # 2 or 3 chunks, the change inside a sequence; ragged vocabulary, padded rows
    (592, 16, 4100, 4104),    # one chunk a row and no row with two
    (576, 64, 4100, 4104),    # one chunk or two
    (593, 593, 2100, 2104),   # more rows than places: equal chunks
    (42, 7, 40001, 40008),    # 14 or 15
    (19, 19, 126464, 126464), # 31 or 32: the most that one CTA finishes
    (18, 6, 126464, 126464),  # 32 or 33: two ticket levels
    (3, 3, 400002, 400008),   # the limit of splits
    (32, 32, 36863, 36864),   # one column short of the smallest chunk: equal chunks
    (32, 32, 38912, 38912),   # the smallest chunk
])
def test_rows_cut_into_unequal_numbers_of_chunks(dtype, R, rps, V, stride):
    d = syn.logits_rows(R, V, dtype, cfg_id=60 + R % 7, row_stride=stride)
    flags = syn.decoded_flags(R, max(1, rps // 2), rps, cfg_id=61)
    o = oracle.entropy_gate(d["logits"], dtype, V, flags, 2.0, rps)
    for _ in range(2):   # (the tickets are zero again)
        _compare(_run_gpu(d["logits"], dtype, V, flags, 2.0, rps), o, 2.0)
