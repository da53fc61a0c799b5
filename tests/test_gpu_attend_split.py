"""16-bit attention in four launches (few groups, or sequences whose K and V do not fit in shared memory) against the
float64 oracle, and its selections against the CTA-per-group kernels bit for bit: every head width, one and many parts of
the keys, lists around the tile edges, tied scores and a NaN row."""
import pytest
import torch

import paper_2604_08971_b200 as sentry
import synth
from tests import parity
from tests.parity import TOL

pytestmark = pytest.mark.gpu


def n_s_of(tv):
    return sentry.num_active_queries(tv, 5)


def _w(name, dtype, B, lengths, Hq, Hk, d, k_h, rule="cycle7"):
    return synth.Workload(name, dtype, B, lengths, 64, Hq, Hk, d, 128, k_h, 64, rule, 11 + d)


@pytest.mark.parametrize("w", [
    _w("split_d16_one_present", "bf16", 16, (1, 510, 1), 4, 1, 16, 3),            # T_v = 1 and 2 in some samples
    _w("split_d16_parts", "bf16", 9, (1400, 1300, 1396), 8, 2, 16, 5),            # T = 4096, 16 keys each lane to select from
    _w("split_d32_tile_edges", "bf16", 8, (127, 257, 129), 6, 2, 32, 4),          # score blocks of 128 end at each list's edge
    _w("split_d32_f16", "f16", 16, (384, 385, 255), 8, 2, 32, 8, "all"),          # every head kept
    _w("split_d32_long", "bf16", 2, (3000, 2500, 2500), 4, 1, 32, 2, "all"),      # T = 8000: 16 parts
    _w("split_d64_few", "f16", 8, (100, 99, 57), 8, 4, 64, 3),                    # T = 256: one part
    _w("split_d64_wide", "bf16", 70, (300, 200, 203), 4, 2, 64, 2),               # a warp per head to select
], ids=lambda w: w.name)
def test_four_launch_attention(w):
    sn = sentry.Sentry(0)
    try:
        inp = synth.generate(w, n_s_of)
        kept_h, _ = parity.gate_lists(sn, inp)
        for mode in (0, 1) if w.T <= 1024 else (0,):
            err, _ = parity.attend_parity(sn, inp, kept_h, None if w.B < 20 else range(0, w.B, 9), mode, full_batch=True)
            assert err <= TOL[w.dtype], (w.name, mode, err)
        ids, masks = parity.dev(inp.ids), parity.masks_dev(inp.masks)
        tbl, offs = parity.dev(inp.sample_table), parity.dev(inp.table_offsets)
        Q, K, V = inp.Q.cuda(), inp.K.cuda(), inp.V.cuda()
        Q[0, :, 7:40] = Q[0, :, 7:8]      # equal queries, and below equal keys: ties at the threshold
        K[0, :, 3:] = K[0, :, 3:4]
        Q[1, 0, 5] = float("nan")
        args = (Q, K, V, kept_h, ids, masks, tbl, offs)
        O, act = sn.attend_fwd(*args, c=w.c, return_active=True)
        assert sn.last_launch_count() == 4
        sn.set_attend_kernel(sentry.ATTEND_WARP_MMA)
        O1, act1 = sn.attend_fwd(*args, c=w.c, return_active=True)
        assert torch.equal(act, act1)
        assert torch.equal(O.isnan(), O1.isnan())
        a, b = torch.nan_to_num(O.float()), torch.nan_to_num(O1.float())
        assert (a - b).abs().max().item() <= TOL[w.dtype] * b.abs().max().item()
        # the same rows given by the caller
        sn.set_attend_kernel(sentry.ATTEND_AUTO)
        O2 = sn.attend_fwd(*args, c=w.c, active_in=act)
        assert torch.equal(torch.nan_to_num(O2.float()), torch.nan_to_num(O.float()))
    finally:
        sn.close()


@pytest.mark.parametrize("w", [
    _w("split_common_d16", "bf16", 30, (342, 341, 341), 8, 2, 16, 8, "all"),
    _w("split_common_d32", "bf16", 16, (342, 341, 341), 8, 2, 32, 4, "all"),
    _w("split_common_d32_f16", "f16", 16, (342, 341, 341), 8, 2, 32, 8, "all"),
    _w("split_common_d64", "bf16", 16, (100, 100, 100), 8, 2, 64, 8, "all"),
], ids=lambda w: w.name)
def test_selection_does_not_depend_on_the_form(w):
    """Keys with a large common part: the raw scores are 2^10 times what is ranked, and so is their rounding.  The lists are
    those of the one-launch form's fp32 loop all the same."""
    sn = sentry.Sentry(0)
    try:
        inp = synth.generate(w, n_s_of)
        kept_h, _ = parity.gate_lists(sn, inp)
        ids, masks = parity.dev(inp.ids), parity.masks_dev(inp.masks)
        tbl, offs = parity.dev(inp.sample_table), parity.dev(inp.table_offsets)
        Q, V = inp.Q.cuda(), inp.V.cuda()
        for power in (8, 13, 15):
            K = inp.K.cuda()
            K[..., 0] = 2.0 ** power
            for mode in (0, 1):
                act = []
                for kernel, launches in ((sentry.ATTEND_AUTO, 4), (sentry.ATTEND_WARP_MMA, 1)):
                    sn.set_attend_kernel(kernel)
                    act.append(sn.attend_fwd(Q, K, V, kept_h, ids, masks, tbl, offs, c=w.c, score_mode=mode, return_active=True)[1])
                    assert sn.last_launch_count() == launches
                assert torch.equal(act[0], act[1]), (w.name, power, mode)
    finally:
        sn.close()


def test_tied_scores_take_no_longer():
    """Zero queries (a padded window): every score of a list ties.  The time of a call does not depend on the values; the bound
    is twice the time of normal data, where a path for ties that scores entries one by one takes nine times as long."""
    w = _w("split_tied", "bf16", 16, (1366, 1365, 1365), 8, 2, 32, 4, "all")
    sn = sentry.Sentry(0)
    try:
        inp = synth.generate(w, n_s_of)
        kept_h, _ = parity.gate_lists(sn, inp)
        args = (kept_h, parity.dev(inp.ids), parity.masks_dev(inp.masks), parity.dev(inp.sample_table), parity.dev(inp.table_offsets))
        Q, K, V = inp.Q.cuda(), inp.K.cuda(), inp.V.cuda()
        O = torch.empty((w.B, w.k_h, w.T, w.d), dtype=Q.dtype, device="cuda")

        def best_ms(q):
            best = float("inf")
            for _ in range(5):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                for _ in range(10):
                    sn.attend_fwd(q, K, V, *args, c=w.c, O=O)
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b))
            return best
        zero = torch.zeros_like(Q)
        act = sn.attend_fwd(zero, K, V, *args, c=w.c, return_active=True)[1]
        assert sn.last_launch_count() == 4
        assert torch.equal(act.cpu(), torch.arange(n_s_of(w.T)).int().expand_as(act))   # ties: the first U
        assert best_ms(zero) <= 2 * best_ms(Q)
    finally:
        sn.close()


@pytest.mark.parametrize("w, launches", [
    (_w("form_96_heads_d32", "bf16", 4, (86, 85, 85), 96, 24, 32, 48), 1),     # 96 groups whose K and V fit: one launch
    (_w("form_96_heads_d16", "f16", 8, (171, 171, 170), 96, 24, 16, 40), 1),
    (_w("form_96_heads_few", "bf16", 1, (171, 171, 170), 96, 24, 32, 48, "all"), 4),
], ids=lambda v: v.name if hasattr(v, "name") else str(v))
def test_the_form_does_not_depend_on_the_number_of_heads(w, launches):
    sn = sentry.Sentry(0)
    try:
        inp = synth.generate(w, n_s_of)
        kept_h, _ = parity.gate_lists(sn, inp)
        err, _ = parity.attend_parity(sn, inp, kept_h, None, 0, full_batch=True)
        assert sn.last_launch_count() == launches
        assert err <= TOL[w.dtype]
    finally:
        sn.close()


@pytest.mark.parametrize("mode", [0, 1, 2])
def test_odd_inputs_are_treated_as_in_one_launch(mode):
    """Token ids that start off a 16-byte boundary and name modalities out of range, a sample without any modality, a subset
    without a table, sampled positions outside the list: the lists, the zero rows and the status word of the other form."""
    w = _w("split_odd", "bf16", 16, (172, 170, 173), 8, 2, 32, 5)
    sn = sentry.Sentry(0)
    try:
        inp = synth.generate(w, n_s_of)
        kept_h, _ = parity.gate_lists(sn, inp)
        ids = torch.empty(w.T + 1, dtype=torch.int32, device="cuda")[1:]
        ids.copy_(parity.dev(inp.ids))
        masks = parity.masks_dev(inp.masks)
        tv = [int(sum(n for j, n in enumerate(w.lengths) if (int(m) >> j) & 1)) for m in inp.masks]
        masks[3] = 0
        offs = parity.dev(inp.table_offsets).clone()
        table = parity.dev(inp.sample_table).clone()
        if mode == 0:
            table[int(offs[int(inp.masks[6])]) + 77] = w.T      # one entry beyond the list, one before it
            table[int(offs[int(inp.masks[5])]) + 5] = -1
        if mode == 2:
            table = parity.dev(synth.entry_major_tables(w, inp.sample_table, inp.table_offsets, n_s_of))
            offs[int(inp.masks[1])] = -1
        if mode == 1:
            ids[10], ids[w.T - 1] = 40, -7                       # present in no sample
        out = []
        for kernel, launches in ((sentry.ATTEND_AUTO, 4), (sentry.ATTEND_WARP_MMA, 1)):
            sn.set_attend_kernel(kernel)
            O, act = sn.attend_fwd(inp.Q.cuda(), inp.K.cuda(), inp.V.cuda(), kept_h, ids, masks, table, offs, c=w.c,
                                   score_mode=mode, return_active=True)
            assert sn.last_launch_count() == launches
            out.append((O.float(), act, sn.last_status()))
        (O, act, status), (O1, act1, status1) = out
        assert torch.equal(act, act1) and status == status1 != 0
        assert O[3].abs().max().item() == 0 and (act[3] == -1).all()
        assert (O - O1).abs().max().item() <= TOL[w.dtype] * O1.abs().max().item()
        assert tv[6] == w.T
    finally:
        sn.close()
