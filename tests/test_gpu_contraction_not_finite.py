"""Rotations and separations that are not finite, or whose length overflows, in the contraction: the item
gives NaN (energy, force and torques), as double arithmetic has it, and its neighbours keep their bits.
Few and many items (descriptors made on the host and on the device), B rotated from its cache (phases of
the rotation), and R0 infinite (phases of the frame).  At degree 0 nothing is rotated: the energy
keeps its value."""
import numpy as np
import pytest
import torch

from paper_0704_1672_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [3, 200])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_phases_that_are_not_finite(precision, k):
    from paper_0704_1672_gb300 import build
    build.build()
    from paper_0704_1672_gb300 import tcm
    prec = tcm.TCM_FP64 if precision == "fp64" else tcm.TCM_MIXED
    rng = np.random.default_rng(k)
    A, B = (torch.tensor(synth.pack(synth.uniform_ball(rng, n, 4.0), rng.normal(size=n)), device="cuda") for n in (150, 120))
    rot = synth.random_rotations(rng, k)
    R0 = synth.unit_vectors(rng, k) * 20.0
    a, b = np.zeros(k, int), np.ones(k, int)
    with tcm.Context(lmax_cap=24) as ctx:
        m = [ctx.tcm_moments(x, 12, precision=prec) for x in (A, B)]
        systems = [tcm.make_system(x, q.center, q.radius, moments=q) for x, q in zip((A, B), m)]
        ctx.tcm_ctx_set_rotate_cached(True)

        def run(L, rot, R0):
            E, _ = ctx.tcm_energy_batch(systems, a, b, np.full(k, L), R0, rotB=rot, precision=prec)
            Eg, G, st = ctx.tcm_gradients_batch(systems, a, b, np.full(k, L), R0, rotB=rot, precision=prec)
            torch.cuda.synchronize()
            assert bool(torch.all(st == 0)) and torch.equal(E.nan_to_num(7.0), Eg.nan_to_num(7.0))
            return E.cpu().numpy(), G.cpu().numpy()

        others = np.arange(k) != 1
        for L in (1, 12):
            E0, G0 = run(L, rot, R0)
            assert np.all(np.isfinite(E0)) and np.all(np.isfinite(G0))
            for entry in range(9):
                for v in (np.nan, np.inf):
                    bad = rot.copy()
                    bad[1].flat[entry] = v
                    E, G = run(L, bad, R0)
                    assert np.isnan(E[1]) and np.all(np.isnan(G[1])), (L, entry, v, E[1])
                    assert np.array_equal(E[others], E0[others]) and np.array_equal(G[others], G0[others])
            for R in ([np.inf, 0.0, 0.0], [1.0, -np.inf, 2.0], [1e200, 0.0, 0.0]):
                far = R0.copy()
                far[1] = R
                E, G = run(L, rot, far)
                assert np.isnan(E[1]) and np.all(np.isnan(G[1])), (L, R, E[1])
                assert np.array_equal(E[others], E0[others]) and np.array_equal(G[others], G0[others])
        E0, _ = run(0, rot, R0)
        bad = rot.copy()
        bad[1, 0, 0] = np.nan
        E, _ = run(0, bad, R0)
        assert np.array_equal(E, E0)
