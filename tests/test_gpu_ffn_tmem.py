"""The fused FFN with the hidden tile in tensor memory (16-bit, d_model 128 and 256) where its tiles can go wrong: last chunks of
every width, one row, lists with odd and even numbers of row tiles, more tiles than CTAs, and the pairs of CTAs that large
calls take, whose results are the single CTAs' to the bit."""
import numpy as np
import pytest
import torch

import paper_2604_08971_b200 as sentry
import synth
from tests import parity
from tests.parity import TOL

pytestmark = pytest.mark.gpu


def _w(name, dtype, B, lengths, D, F, k_c, rule="cycle7"):
    return synth.Workload(name, dtype, B, lengths, D, 4, 2, 16, F, 2, k_c, rule, 7, w_std=0.05)


@pytest.mark.parametrize("D,k_c", [(D, k) for D in (128, 256) for k in (1, 63, 64, 65, 127, 128, 129, 192, 193, 256, 330)])
def test_last_chunk(D, k_c):
    w = _w("tmem_d%d_k%d" % (D, k_c), "f16" if k_c % 2 else "bf16", 7, (61, 50, 37), D, 384, k_c)
    sn = sentry.Sentry(0)
    try:
        inp = synth.generate(w, lambda tv: sentry.num_active_queries(tv, 5))
        _, kept_c = parity.gate_lists(sn, inp)
        # The bound is for sums of many channels, whose errors (a hidden value is off by up to 2^-11 of the tanh unit, 1.5e-4
        # of its fit and half an ulp of the storage: 9e-4 for half) average out.  A single channel's result is off by that
        # share of ITS OWN size, and the largest of the call's 76 k products of two normals is about 13 RMS: 1.2e-2.
        assert parity.ffn_parity(sn, inp, kept_c) <= TOL[w.dtype] * (3 if k_c == 1 else 1)
    finally:
        sn.close()


@pytest.mark.parametrize("D", [128, 256])
def test_one_row(D):
    w = _w("tmem_d%d_one_row" % D, "bf16", 1, (1, 1, 1), D, 256, 40)
    sn = sentry.Sentry(0)
    try:
        inp = synth.generate(w, lambda tv: sentry.num_active_queries(tv, 5))
        _, kept_c = parity.gate_lists(sn, inp)
        assert parity.ffn_parity(sn, inp, kept_c) <= TOL["bf16"]
    finally:
        sn.close()


# kept channels, lists, samples, element type; with 148 SMs all but the first go to pairs (tests/test_ffn_pair_rule.py holds them to that)
PAIRS = [(65, 7, 1280, "bf16"), (200, 3, 1800, "bf16"), (384, 1, 1280, "bf16"), (130, 64, 1800, "bf16"), (512, 7, 900, "bf16"),
         (512, 1, 640, "bf16"), (129, 5, 1900, "f16"), (257, 1, 900, "f16"), (512, 7, 900, "f16")]
PAIR_T, PAIR_STEP = 100, 160


@pytest.mark.parametrize("k_c,n_lists,B,dtype", PAIRS)
def test_pairs_equal_single_ctas(k_c, n_lists, B, dtype):
    """A large call (pairs of CTAs where there is more than one chunk of 128 channels) against the same samples in small calls
    (single CTAs): equal bits, and equal again."""
    gen = torch.Generator(device="cuda").manual_seed(k_c)
    T, D, F = PAIR_T, 256, 512
    dt = torch.bfloat16 if dtype == "bf16" else torch.float16
    X = torch.randn((B, T, D), generator=gen, device="cuda").to(dt)
    W1 = torch.randn((D, F), generator=gen, device="cuda").mul_(0.05).to(dt)
    W2 = torch.randn((F, D), generator=gen, device="cuda").mul_(0.05).to(dt)
    u = torch.rand((n_lists, F), generator=gen, device="cuda")
    kept = u.topk(k_c, dim=1).indices.sort(dim=1).values.int().contiguous()
    ids = torch.tensor([0] * 41 + [1] * 33 + [2] * 26, dtype=torch.int32, device="cuda")
    rng = np.random.default_rng(k_c)
    masks = torch.from_numpy(rng.integers(1, 8, B).astype(np.int32)).cuda()
    lists = torch.from_numpy(rng.integers(0, n_lists, B).astype(np.int32)).cuda()
    sn = sentry.Sentry(0)
    try:
        Y = sn.ffn_fwd(X, W1, W2, kept, lists, ids, masks)
        assert torch.equal(Y, sn.ffn_fwd(X, W1, W2, kept, lists, ids, masks))
        step = PAIR_STEP
        for b in range(0, B, step):
            part = sn.ffn_fwd(X[b:b + step].contiguous(), W1, W2, kept, lists[b:b + step].contiguous(), ids, masks[b:b + step].contiguous())
            assert torch.equal(Y[b:b + step], part)
        assert sn.last_status() == 0
    finally:
        sn.close()
