"""The one-launch attention where its token list, its head list, its score loop and its selections can go wrong, against the
float64 oracle: one to five tokens, counts of sampled keys of every remainder, lists around the edges of a round of counts, more than
32 kept heads, groups of four heads in one pass and (many waves of CTAs) in two, and scores that tie."""
import numpy as np
import pytest
import torch

import paper_2604_08971_b200 as sentry
import synth
from tests import parity
from tests.parity import TOL

pytestmark = pytest.mark.gpu


def n_s_of(tv):
    return sentry.num_active_queries(tv, 5)


def _w(name, dtype, B, lengths, Hq, Hk, d, k_h, rule="cycle7", c=5):
    return synth.Workload(name, dtype, B, lengths, 64, Hq, Hk, d, 64, k_h, 8, rule, 11, c=c)


@pytest.fixture
def sn():
    s = sentry.Sentry(0)
    s.set_attend_kernel(sentry.ATTEND_WARP_MMA)
    yield s
    s.close()


@pytest.mark.parametrize("w", [
    _w("fused_few_tokens", "bf16", 7, (1, 2, 2), 8, 2, 32, 5),
    _w("fused_counts_mod4", "bf16", 21, (3, 8, 30), 8, 4, 16, 6, c=3),
    _w("fused_round_edge_128", "f16", 7, (1, 127, 128), 8, 2, 32, 8),                # T = 256: two rounds of 128 threads
    _w("fused_round_edge_256", "bf16", 7, (256, 1, 255), 6, 2, 32, 6),               # T = 512 on 256 threads
    _w("fused_two_count_rounds", "bf16", 3, (1024, 1025, 251), 4, 2, 16, 4, "all"),  # T = 2300 > 4 x 512
    _w("fused_48_heads", "bf16", 4, (20, 11, 9), 64, 16, 16, 48),
    _w("fused_many_waves", "bf16", 640, (5, 6, 9), 16, 4, 32, 16),                   # 2560 CTAs, four heads to a group
    _w("fused_one_wave_of_fours", "bf16", 20, (50, 60, 90), 16, 4, 32, 16),
    _w("fused_d64", "f16", 9, (64, 65, 66), 8, 2, 64, 7),
], ids=lambda w: w.name)
@pytest.mark.parametrize("arranged", [False, True])
def test_matches_oracle(sn, w, arranged):
    inp = synth.generate(w, n_s_of)
    kept_h, _ = parity.gate_lists(sn, inp)
    samples = None if w.B <= 64 else np.arange(0, w.B, 37)
    err, _ = parity.attend_parity(sn, inp, kept_h, samples=samples, full_batch=True, arranged=arranged)
    assert sn.last_launch_count() == 1 and err <= TOL[w.dtype]


@pytest.mark.parametrize("T,B", [(200, 4), (700, 4), (1000, 4), (200, 2600)])
@pytest.mark.parametrize("zero", ["all", "half", "few"])
def test_ties_go_to_the_lower_position(sn, T, B, zero):
    """Zero queries score 0 whatever their keys, the others above 0 (a maximum lies above its mean): the list is known without
    computing a score."""
    w = _w("fused_ties", "bf16", B, (T, 0, 0), 4, 1, 32, 4, "all")
    inp = synth.generate(w, n_s_of)
    kept_h, _ = parity.gate_lists(sn, inp)
    U = n_s_of(T)
    Q = inp.Q.cuda().clone()
    top = torch.arange(3, T, 11, device="cuda")[: U // 2]          # positions that keep their queries
    if zero == "all":
        Q.zero_()
        want = torch.arange(U)
    elif zero == "half":                                            # U positions with a score, all others tie at 0
        keep = torch.arange(0, T, max(1, T // U), device="cuda")[:U]
        mask = torch.ones(T, dtype=torch.bool, device="cuda")
        mask[keep] = False
        Q[:, :, mask] = 0
        want = keep.cpu()
    else:
        mask = torch.ones(T, dtype=torch.bool, device="cuda")
        mask[top] = False
        Q[:, :, mask] = 0
        rest = [t for t in range(T) if t not in set(top.tolist())][: U - len(top)]
        want = torch.tensor(sorted(top.tolist() + rest))
    act = sn.attend_fwd(Q, inp.K.cuda(), inp.V.cuda(), kept_h, parity.dev(inp.ids), parity.masks_dev(inp.masks),
                        parity.dev(inp.sample_table), parity.dev(inp.table_offsets), c=w.c, return_active=True)[1]
    assert sn.last_launch_count() == 1 and sn.last_status() == 0
    assert torch.equal(act.cpu(), want.int().expand_as(act.cpu()))
