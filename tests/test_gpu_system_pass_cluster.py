"""Systems on one cluster of eight CTAs of which some own no atoms (1,025 double records fill five; eight
are started): those reach the exchange through distributed shared memory at once, and must not
before every CTA of the cluster has started.  Many copies of such systems in one call, more clusters than
are resident together, each with the bits of a call of its own; centre computed and given.  The values
themselves are compared with the oracle in test_gpu_system_pass.py."""
import numpy as np
import pytest
import torch

from paper_0704_1672_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("n, dtype", [(1025, torch.float64), (1290, torch.float64), (8193, torch.float32)])
def test_copies_in_one_call_have_the_bits_of_one(n, dtype, given):
    from paper_0704_1672_gb300 import build
    build.build()
    from paper_0704_1672_gb300 import tcm
    rng = np.random.default_rng(n)
    X = torch.tensor(synth.pack(synth.uniform_ball(rng, n, 20.0), rng.normal(size=n)), dtype=dtype, device="cuda")
    c = np.array([0.5, -0.25, 0.125]) if given else None
    k = 640
    R0 = np.tile([[0.0, 36.0, 48.0]], (k, 1))
    with tcm.Context(lmax_cap=4) as ctx:
        E1, s1 = ctx.tcm_energy_batch([(X, c, None)] * 2, [0], [1], [2], R0[:1])
        for _ in range(5):
            Y = [X.clone() for _ in range(k)]
            E, s = ctx.tcm_energy_batch([(y, c, None) for y in Y], np.arange(k), (np.arange(k) + 1) % k, np.full(k, 2), R0)
            torch.cuda.synchronize()
            assert int(s1[0]) == 0 and bool(torch.all(s == 0))
            assert bool(torch.all(E == E1[0]))
