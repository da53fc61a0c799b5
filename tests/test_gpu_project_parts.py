"""The tensor-core projections where their tiles can go wrong, against the float64 oracle: one and several parts of the
output columns, tiles that end half way, one token, more heads than a stage ring holds, every head width; and the plain-ALU ones with
as many slices as there can be."""
import numpy as np
import pytest
import torch

import oracle
import paper_2604_08971_b200 as sentry
import synth
from tests import parity
from tests.parity import TOL, dev, masks_dev

pytestmark = pytest.mark.gpu


def n_s_of(tv):
    return sentry.num_active_queries(tv, 5)


def _w(name, dtype, B, lengths, D, Hq, Hk, d, k_h, rule="cycle7"):
    return synth.Workload(name, dtype, B, lengths, D, Hq, Hk, d, 128, k_h, 64, rule, 5 + d)


@pytest.mark.parametrize("w", [
    _w("parts_d16_one_token", "bf16", 3, (1, 1, 1), 64, 2, 1, 16, 1),
    _w("parts_d16_24_slices", "bf16", 7, (63, 64, 130), 128, 24, 4, 16, 18),      # 26 slices in two parts of 13
    _w("parts_d32_3_parts", "f16", 7, (127, 2, 129), 256, 16, 8, 32, 9),          # 9 + up to 16 slices: up to four parts
    _w("parts_d64_5_slices", "bf16", 5, (40, 128, 88), 128, 6, 2, 64, 3),         # parts of 3 and 2 or 4 and 3 slices
    _w("parts_d64_wide_out", "bf16", 4, (200, 97, 90), 768, 12, 4, 64, 7, "all"),    # output in three parts; plain-ALU Q, K, V
    _w("parts_d16_2000_tokens", "bf16", 7, (1500, 37, 460), 64, 4, 2, 16, 3),     # a warp's run of token pieces above eight; empty tiles
    _w("plain_f32_128_slices", "f32", 2, (5, 6, 7), 64, 64, 32, 16, 64),          # 64 heads, K and V of 32 groups
    _w("plain_f32_40_of_48", "f32", 3, (5, 6, 7), 320, 48, 12, 16, 40),           # list entries beyond a warp's first 32
    _w("parts_d32_wide_out", "f16", 4, (30, 97, 90), 320, 12, 4, 32, 12),         # five column boxes in parts of 3 and 2
], ids=lambda w: w.name)
def test_projection_parts(w):
    sn = sentry.Sentry(0)
    try:
        inp = synth.generate(w, n_s_of)
        kept_h, _ = parity.gate_lists(sn, inp)
        g = torch.Generator().manual_seed(w.seed)
        dt = synth.torch_dtype(w)
        WQ, WK, WV, WO = ((torch.randn(s, generator=g) * 0.08).to(dt) for s in (
            (w.D, w.Hq * w.d), (w.D, w.Hk * w.d), (w.D, w.Hk * w.d), (w.Hq * w.d, w.D)))
        ids, masks = dev(inp.ids), masks_dev(inp.masks)
        Q, K, V = (torch.full((w.B, H, w.T, w.d), 7.0, dtype=dt, device="cuda") for H in (w.Hq, w.Hk, w.Hk))
        sn.project_qkv(inp.X.cuda(), WQ.cuda(), WK.cuda(), WV.cuda(), kept_h, ids, masks, w.Hq, w.Hk, w.d, Q=Q, K=K, V=V)
        kh = kept_h.cpu().numpy()
        present = ((inp.masks[:, None].astype(np.int64) >> inp.ids[None, :]) & 1).astype(bool)
        want = oracle.project_qkv(inp.X, WQ, WK, WV, kh, inp.ids, inp.masks, w.Hq, w.Hk, w.d)
        for got_t, want_t, heads in ((Q, want[0], kh), (K, want[1], kh // (w.Hq // w.Hk)), (V, want[2], kh // (w.Hq // w.Hk))):
            got, written = got_t.float().cpu().numpy(), np.zeros(got_t.shape[:3], dtype=bool)
            for b in range(w.B):
                written[b][np.ix_(np.unique(heads[b]), np.nonzero(present[b])[0])] = True
            assert np.all(got[~written] == 7.0)
            assert parity.rel_err(got[written], want_t[written], w.dtype, np.ones(int(written.sum()), dtype=bool)) <= TOL[w.dtype]
        A = (torch.randn((w.B, w.k_h, w.T, w.d), generator=g)).to(dt)
        out = sn.project_out(A.cuda(), WO.cuda(), kept_h, ids, masks, w.Hq, out=torch.full((w.B, w.T, w.D), 7.0, dtype=dt, device="cuda"))
        assert sn.last_status() == 0
        got = out.float().cpu().numpy()
        assert np.all(got[~present] == 0.0)
        want_out = oracle.project_out(A, WO, kh, inp.ids, inp.masks, w.Hq)
        assert parity.rel_err(got, want_out, w.dtype, np.ones(got.shape[:2], dtype=bool)) <= TOL[w.dtype]
    finally:
        sn.close()
