"""The plain-ALU kernels against the float64 oracle where their pieces end: FFN tiles of 4 and of 16 rows around the row
count that separates them, d_model in one and in several 256-column pieces, channel counts around a piece; attention with
its rows in many parts and in one."""
import pytest

import paper_2604_08971_b200 as sentry
import synth
from tests import parity
from tests.parity import TOL

pytestmark = pytest.mark.gpu


def n_s_of(tv):
    return sentry.num_active_queries(tv, 5)


@pytest.mark.parametrize("w", [
    synth.Workload("alu_one_row", "f32", 1, (1, 1, 1), 8, 2, 1, 16, 16, 1, 1, "cycle7", 3),
    synth.Workload("alu_592_rows", "f32", 4, (74, 74), 64, 4, 2, 32, 300, 3, 257, "all", 4),
    synth.Workload("alu_596_rows", "f32", 4, (75, 74), 64, 4, 2, 32, 300, 3, 256, "all", 5),
    synth.Workload("alu_d264", "f32", 7, (9, 3, 30), 264, 6, 3, 64, 64, 4, 41, "cycle7", 6),
    synth.Workload("alu_d1000_f16", "f16", 3, (9, 3, 3), 1000, 4, 2, 16, 64, 2, 9, "cycle7", 7),
    synth.Workload("alu_many_samples", "f32", 150, (20, 15), 72, 4, 2, 16, 64, 3, 24, "dropout0.3", 8),
], ids=lambda w: w.name)
def test_plain_alu_kernels(w):
    sn = sentry.Sentry(0)
    try:
        inp = synth.generate(w, n_s_of)
        kept_h, kept_c = parity.gate_lists(sn, inp)
        assert parity.attend_parity(sn, inp, kept_h)[0] <= TOL[w.dtype]
        assert parity.ffn_parity(sn, inp, kept_c) <= TOL[w.dtype]
    finally:
        sn.close()
