"""The channel-compacted FFN as two tensor-core GEMMs (d_model a multiple of 64 other than 128, 256, 384) against the
float64 oracle, where its tiles can go wrong: one K block, column tiles that end half way, ragged channel counts, row
tiles of several lists, more row tiles than the hidden buffer holds, and as the experts' FFN of a Sparse-MoE block."""
import numpy as np
import pytest
import torch

import oracle
import paper_2604_08971_b200 as sentry
import synth
from tests import parity
from tests.parity import TOL

pytestmark = pytest.mark.gpu


def n_s_of(tv):
    return sentry.num_active_queries(tv, 5)


def _w(name, dtype, B, lengths, D, F, k_c, rule="cycle7"):
    return synth.Workload(name, dtype, B, lengths, D, 4, 2, 16, F, 2, k_c, rule, 7, w_std=0.05)


@pytest.mark.parametrize("w", [
    _w("wide_d64_one_row", "bf16", 1, (1, 1, 1), 64, 128, 8),
    _w("wide_d192_ragged", "bf16", 9, (37, 5, 91), 192, 400, 201),
    _w("wide_d768_lists", "bf16", 8, (61, 47, 20), 768, 1024, 300),
    _w("wide_d1024_f16", "f16", 3, (40, 50, 39), 1024, 512, 129),
    _w("wide_d320_turns", "bf16", 70, (100, 100, 100), 320, 256, 128, "all"),   # 165 row tiles: two turns of the buffer
], ids=lambda w: w.name)
def test_wide_ffn_matches_oracle(w):
    sn = sentry.Sentry(0)
    try:
        inp = synth.generate(w, n_s_of)
        _, kept_c = parity.gate_lists(sn, inp)
        assert parity.ffn_parity(sn, inp, kept_c) <= TOL[w.dtype]
        # materialised once: the same bits, and the same again
        los, ids, masks = (parity.dev(inp.list_of_sample), parity.dev(inp.ids), parity.masks_dev(inp.masks))
        X, W1, W2 = inp.X.cuda(), inp.W1.cuda(), inp.W2.cuda()
        Y = sn.ffn_fwd(X, W1, W2, kept_c, los, ids, masks)
        packed = sn.ffn_prepack(W1, W2, kept_c)
        Y2 = sn.ffn_fwd_packed(X, packed, w.F, w.k_c, kept_c.shape[0], los, ids, masks)
        assert torch.equal(Y, Y2) and sn.last_status() == 0
    finally:
        sn.close()


@pytest.mark.parametrize("dtype,large", [("bf16", (2.0e38, -2.0e38, 3.38e38, -3.38e38, 1.0e30)), ("f16", (60000.0, -60000.0, 40000.0))])
def test_wide_ffn_extreme_values(dtype, large):
    """One channel a column (W1, W2 the identity), so that a pre-activation is X's value: large finite ones come back
    (gelu(z) = z, or 0 below), an infinite or NaN one spoils its own row and no other."""
    dt = torch.bfloat16 if dtype == "bf16" else torch.float16
    D, T = 64, 130
    X = torch.randn((1, T, D), generator=torch.Generator().manual_seed(1)).to(dt)
    special = {}
    for i, v in enumerate(large + (float("inf"), float("-inf"), float("nan"))):
        X[0, 7 * i + 3, i] = v
        special[7 * i + 3] = v
    eye, kept = torch.eye(D).to(dt), torch.arange(D, dtype=torch.int32).reshape(1, D)
    sn = sentry.Sentry(0)
    try:
        Y = sn.ffn_fwd(X.cuda(), eye.cuda(), eye.cuda(), kept.cuda(), torch.zeros(1, dtype=torch.int32).cuda()).cpu()[0]
        want = torch.nn.functional.gelu(X[0].double())
        for r in range(T):
            if np.isfinite(special.get(r, 0.0)):   # (the two roundings of a stored value, and fp32 sums)
                assert torch.allclose(Y[r].double(), want[r], rtol=2.0 ** (-8 if dtype == "bf16" else -11) * 1.01, atol=1e-6), r
            else:
                assert not torch.isfinite(Y[r]).all(), r
        assert sn.last_status() == 0
    finally:
        sn.close()


@pytest.mark.parametrize("dtype,x,scale", [("f16", 60000.0, 2.0), ("f16", -60000.0, 2.0), ("f16", 65504.0, 1.0), ("bf16", 3.38e38, 1.0078125)])
def test_wide_ffn_hidden_value_beyond_the_storage_type(dtype, x, scale):
    """A hidden value above the largest 16-bit one (below twice it) reaches a result that is in range."""
    dt = torch.bfloat16 if dtype == "bf16" else torch.float16
    D = 64
    X = torch.randn((1, 3, D), generator=torch.Generator().manual_seed(2)).to(dt)
    X[0, 1, 5] = x
    W1, W2 = (torch.eye(D) * scale).to(dt), (torch.eye(D) * 0.25).to(dt)
    z = X[0].double() * float(W1[0, 0])
    sn = sentry.Sentry(0)
    try:
        Y = sn.ffn_fwd(X.cuda(), W1.cuda(), W2.cuda(), torch.arange(D, dtype=torch.int32).reshape(1, D).cuda(),
                       torch.zeros(1, dtype=torch.int32).cuda()).cpu()[0]
        want = torch.nn.functional.gelu(z) * 0.25
        assert torch.allclose(Y.double(), want, rtol=2.0 ** (-8 if dtype == "bf16" else -11) * 1.01, atol=1e-6)
    finally:
        sn.close()


# (d_model, kept channels, row tiles): with 148 SMs every width of the column tiles of GEMM 1 and of both forms of GEMM 2, and last
# tiles of 32 to 128 columns (tests/test_ffn_wide_math.py holds the list to that)
WIDTHS = [(64, 100, 1), (64, 300, 33), (192, 100, 99), (192, 300, 60), (320, 100, 40), (320, 129, 99), (320, 300, 40), (192, 300, 75),
          (320, 300, 60), (512, 300, 45), (192, 385, 60), (320, 385, 75), (768, 1229, 33), (640, 500, 59)]


@pytest.mark.parametrize("D,k_c,tiles", WIDTHS)
def test_wide_ffn_tile_widths(D, k_c, tiles):
    """Against the same sums in float64.  A stored hidden value is off by up to 2^-17 of itself (head and remainder), its GELU and
    the fp32 sums by less; the sum of a result's absolute terms is about 0.65 sqrt(k_c) times the results' RMS, twice that
    in the largest rows: 2^-16 sqrt(k_c) RMS, beside the half unit of the stored result."""
    gen = torch.Generator(device="cuda").manual_seed(D + k_c)
    rows, F = tiles * 128 - 37, k_c + 50
    X = torch.randn((1, rows, D), generator=gen, device="cuda").bfloat16()
    W1 = torch.randn((D, F), generator=gen, device="cuda").mul_(D ** -0.5).bfloat16()
    W2 = torch.randn((F, D), generator=gen, device="cuda").mul_(k_c ** -0.5).bfloat16()
    kept = torch.rand((F,), generator=gen, device="cuda").topk(k_c).indices.sort().values
    sn = sentry.Sentry(0)
    try:
        Y = sn.ffn_fwd(X, W1, W2, kept.int().reshape(1, -1).contiguous(), torch.zeros(1, dtype=torch.int32, device="cuda"))
        want = torch.nn.functional.gelu(X[0].double() @ W1.double()[:, kept]) @ W2.double()[kept]
        half_ulp = torch.exp2(torch.floor(torch.log2(want.abs().clamp_min(1e-30))) - 8)
        excess = ((Y[0].double() - want).abs() - half_ulp).clamp_min(0).max()
        assert float(excess) <= 2.0 ** -16 * k_c ** 0.5 * float(want.square().mean().sqrt())
        assert sn.last_status() == 0
    finally:
        sn.close()


def test_wide_moe_matches_oracle():
    m = synth.generate_moe(300, 512, 256, 5, 2, 100, "bf16", seed=3, skew=1.0)
    sn = sentry.Sentry(0)
    try:
        ids, wts = torch.from_numpy(m.expert_ids).cuda(), torch.from_numpy(m.expert_weights).cuda()
        Y = sn.moe_ffn_fwd(m.X.cuda(), ids, wts, W1=m.W1.cuda(), W2=m.W2.cuda(), kept_channels=torch.from_numpy(m.kept).cuda())
        want = oracle.moe_ffn(m.X, m.W1, m.W2, m.kept, m.expert_ids, m.expert_weights)
        assert parity.rel_err(Y.float().cpu().numpy(), want, "bf16", np.ones(300, dtype=bool)) <= TOL["bf16"]
        assert sn.last_status() == 0
    finally:
        sn.close()
