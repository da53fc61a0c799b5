"""The routing plan of large Sparse-MoE calls against the float64 oracle: just past the one-launch plan, a block's share over
several rounds, more experts than threads, and every slot on one expert."""
import numpy as np
import pytest
import torch

import oracle
import paper_2604_08971_b200 as sentry
import synth
from tests import parity
from tests.parity import TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,D,F,E,top_k,k_c,dtype,unrouted", [
    (8193, 8, 16, 3, 1, 8, "f32", 0.0),
    (5003, 128, 128, 300, 3, 40, "bf16", 0.2),
    (9001, 8, 16, 1500, 4, 8, "f32", 0.1),       # 16 blocks of two rounds
    (9001, 64, 64, 1, 1, 16, "f32", 0.5),
], ids=lambda v: str(v))
def test_moe_plan_of_large_calls(N, D, F, E, top_k, k_c, dtype, unrouted):
    m = synth.generate_moe(N, D, F, E, top_k, k_c, dtype, seed=N, skew=1.0, unrouted=unrouted)
    sn = sentry.Sentry(0)
    try:
        Y = sn.moe_ffn_fwd(m.X.cuda(), torch.from_numpy(m.expert_ids).cuda(), torch.from_numpy(m.expert_weights).cuda(),
                           W1=m.W1.cuda(), W2=m.W2.cuda(), kept_channels=torch.from_numpy(m.kept).cuda())
        assert sn.last_status() == 0
        ids, weights = m.expert_ids.copy(), m.expert_weights.astype(np.float64)   # not routed: expert 0 with weight 0
        weights[ids < 0], ids[ids < 0] = 0.0, 0
        want = oracle.moe_ffn(m.X, m.W1, m.W2, m.kept, ids, weights)
        got = Y.float().cpu().numpy()
        assert parity.rel_err(got, want, dtype, np.ones((N,), dtype=bool)) <= TOL[dtype]
    finally:
        sn.close()
