"""Double path, rotated sides of a batch: B's moments from its lab-frame set rotated in the
contraction when the item's matrix is a rotation to rounding, from the transformed atoms otherwise.
Both against the oracle's moments of the transformed atoms at the 1e-12 bar of the double path."""
import numpy as np
import pytest
import torch

import oracle
from paper_0704_1672_gb300 import synth
from tcm_testlib import TOL_FP64, energy_error

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tcm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0704_1672_gb300 import build
    build.build()
    from paper_0704_1672_gb300 import tcm as t
    torch.cuda.set_device(0)
    return t


@pytest.mark.parametrize("cached", [False, True])
@pytest.mark.parametrize("L", [0, 1, 6, 13])
def test_rotated_sides_fp64(tcm, L, cached):
    rng = np.random.default_rng(40 + L)
    A, B = (synth.pack(synth.uniform_ball(rng, n, r) + [2.0, 1.0, -3.0], rng.normal(0.02, 0.3, n))
            for n, r in ((90, 4.0), (70, 3.0)))
    R = synth.random_rotations(rng, 6)
    mats = [R[0], R[1].astype(np.float32).astype(np.float64),  # a rotation rounded to float
            -R[2], R[3] * (1.0 + 1e-14), np.diag([1.0, 2.0, 0.5]) @ R[4], R[5] @ R[0], np.eye(3)]
    k = len(mats)
    R0 = synth.unit_vectors(rng, k) * 14.0
    R0[0] = [0.0, 0.0, -14.0]
    Ad, Bd = torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda")
    (cA, _), (cB, _) = oracle.center_radius(A), oracle.center_radius(B)
    QA = oracle.moments(A, cA, L)
    with tcm.Context(lmax_cap=24) as ctx:
        systems = [(Ad, None, None), (Bd, None, None)]
        if cached:  # caches of mixed precision: for unrotated sides only, unless the caller says otherwise
            m = [ctx.tcm_moments(x.float(), L, precision=tcm.TCM_MIXED) for x in (Ad, Bd)]
            ma = ctx.tcm_moments(Ad, L, precision=tcm.TCM_FP64)
            systems = [tcm.make_system(Ad, ma.center, ma.radius, moments=ma),
                       tcm.make_system(Bd, cB, 4.0, moments=m[1])]
        args = (systems, np.zeros(k, int), np.ones(k, int), np.full(k, L), R0)
        E, st = ctx.tcm_energy_batch(*args, rotB=np.stack(mats), precision=tcm.TCM_FP64)
        E1, _ = ctx.tcm_energy_batch(systems, [0], [1], [L], R0[5:6], rotB=mats[5][None], precision=tcm.TCM_FP64)
        Eg, _, _ = ctx.tcm_gradients_batch(*args, rotB=np.stack(mats), precision=tcm.TCM_FP64)
        torch.cuda.synchronize()
    assert st.tolist() == [0] * k
    assert float(E1[0]) == float(E[5])  # alone as in the batch, which also has items that use the atoms
    assert torch.equal(E, Eg)
    for i, M in enumerate(mats):
        QB = oracle.moments(B, cB, L, rot=M)
        Eo = oracle.tcm_energy(L, QA, QB, R0[i])
        err = energy_error(float(E[i]), Eo, oracle.tcm_blocks(L, QA, QB, R0[i]))
        assert err < TOL_FP64, (i, err)
