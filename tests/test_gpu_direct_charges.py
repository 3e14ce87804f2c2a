"""The direct sum with charges far from 1 (csrc/direct.cu): the fixed-point form scales B's charges by a
range's largest, which has to leave the sum's own scale in the normal numbers; outside it the double form
takes the range.  Tolerance as in test_gpu_direct.py: 2e-15 (1 + (R + a_A + a_B) / r_min) of
sum |q_i q_j| / r_ij."""
import numpy as np
import pytest
import torch

import oracle
from paper_0704_1672_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("length", [1.0, 1e-80, 1e80])
@pytest.mark.parametrize("ea, eb", [(200, -260), (0, -240), (150, -150), (290, -300), (-300, 100), (-200, 250), (10, -155)])
def test_charges_far_from_one(ea, eb, length):
    from paper_0704_1672_gb300 import build
    build.build()
    from paper_0704_1672_gb300 import tcm
    at = eb - np.log10(length)
    if not -285 < at < 285 or not -285 < at + ea < 285:
        pytest.skip("a potential or energy outside the normal numbers")
    rng = np.random.default_rng(1000 + ea - eb)
    A, B = (synth.pack(length * synth.uniform_ball(rng, n, r), s * rng.normal(size=n))
            for n, r, s in ((300, 9.0, 10.0 ** ea), (700, 4.0, 10.0 ** eb)))
    B[600:, 3] = 0.0
    R0 = length * np.array([[0.0, 30.0, 0.0], [12.0, -16.0, 0.0]])
    with tcm.Context(lmax_cap=4) as ctx:
        E = ctx.tcm_direct_batch(torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda"), R0, cA=np.zeros(3),
                                 cB=np.zeros(3)).cpu().numpy()
    for k in range(2):
        # (the oracle in units of its own: products of these charges and lengths stay in range)
        Au, Bu = A.copy(), B.copy()
        Au[:, :3] /= length
        Bu[:, :3] /= length
        ref, scale = oracle.direct(Au, np.zeros(3), Bu, np.zeros(3), R0[k] / length, return_abs=True)
        R = np.linalg.norm(R0[k]) / length
        assert abs(E[k] * length - ref) <= 2e-15 * (1.0 + (R + 13.0) / (R - 13.0)) * scale, (k, E[k] * length, ref)
