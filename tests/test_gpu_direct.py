"""The two forms of the direct sum's pair loop (csrc/direct.cu): 64-bit fixed point for separated
systems, double for the rest, each against the oracle at the edges of its range.

Tolerance, of sum |q_i q_j| / r_ij: each distance carries the rounding of B's placed position (about
four roundings of R + a_B) and each term and partial sum a few roundings of its own, in the library
and in the oracle alike: 2e-15 (1 + (R + a_A + a_B) / r_min)."""
import numpy as np
import pytest
import torch

import oracle
from paper_0704_1672_gb300 import synth

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


@pytest.fixture(scope="module")
def ctx(tcm):
    c = tcm.Context(lmax_cap=4)
    yield c
    c.close()


def _system(rng, n, radius, scale=1.0):
    S = synth.pack(synth.uniform_ball(rng, n, radius), rng.normal(0.0, 0.3, n))
    S[:, :3] = (S[:, :3] + [3.0, -7.0, 2.0]) * scale
    return S


def _check(ctx, A, B, factors, dtype, rot=None, given=None):
    """Energies at R = factor (a_A + a_B) along fixed directions against the oracle."""
    Ad, Bd = torch.tensor(A, dtype=dtype, device="cuda"), torch.tensor(B, dtype=dtype, device="cuda")
    A, B = Ad.double().cpu().numpy(), Bd.double().cpu().numpy()
    (cA, aA), (cB, aB) = oracle.center_radius(A), oracle.center_radius(B)
    rng = np.random.default_rng(len(A) * 7 + len(B))
    R0 = synth.unit_vectors(rng, len(factors)) * (np.asarray(factors) * (aA + aB))[:, None]
    centers = {} if given is None else {"cA": cA, "cB": cB}
    E = ctx.tcm_direct_batch(Ad, Bd, R0, rotB=rot, **centers)
    torch.cuda.synchronize()
    for k, f in enumerate(factors):
        ref, scale = oracle.direct(A, cA, B, cB, R0[k], rotB=None if rot is None else rot[k], return_abs=True)
        sep = max(f - 1.0, 1e-3)
        tol = 2e-15 * (1.0 + (f + 1.0) / sep) * scale
        assert abs(float(E[k]) - ref) <= tol, (f, float(E[k]), ref, tol)
    return E


FACTORS = [1.02, 1.04, 1.07, 1.2, 1.5, 3.0, 40.0]  # the fixed-point range begins between 1.03 and 1.07


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("na, nb", [(1, 1), (2, 31), (33, 32), (255, 257), (256, 511), (257, 1024), (513, 1025), (700, 40)])
def test_direct_sizes_and_separations(ctx, na, nb, dtype):
    rng = np.random.default_rng(na * 1000 + nb)
    rot = synth.random_rotations(rng, len(FACTORS))
    A, B = _system(rng, na, 9.0), _system(rng, nb, 4.0)
    if na == 1 and nb == 1:  # both radii are zero: any separation is separated
        Ad, Bd = torch.tensor(A, dtype=dtype, device="cuda"), torch.tensor(B, dtype=dtype, device="cuda")
        E = ctx.tcm_direct_batch(Ad, Bd, [[0.0, 3.0, 4.0]])
        q = float(Ad[0, 3]) * float(Bd[0, 3])
        assert abs(float(E[0]) - q / 5.0) <= 4e-16 * abs(q)
        return
    _check(ctx, A, B, FACTORS, dtype, rot=rot)


@pytest.mark.parametrize("scale", [1e-10, 1e9])
def test_direct_scales_charges_and_given_centres(ctx, scale):
    rng = np.random.default_rng(8)
    A, B = _system(rng, 300, 9.0, scale), _system(rng, 600, 4.0, scale)
    B[:, 3] *= 10.0 ** rng.uniform(-8, 8, 600)  # charges over sixteen orders of magnitude
    B[5, 3] = 0.0
    _check(ctx, A, B, FACTORS, torch.float64)
    _check(ctx, A, B, FACTORS, torch.float64, given=True)  # the centre given, no radius
    B[:, 3] = 0.0
    assert torch.all(_check(ctx, A, B, [1.5], torch.float64) == 0)


def test_direct_item_is_the_same_in_any_batch(ctx):
    rng = np.random.default_rng(9)
    A, B = (torch.tensor(_system(rng, n, 6.0), device="cuda") for n in (700, 1300))
    R0 = synth.unit_vectors(rng, 70000) * 40.0
    E = ctx.tcm_direct_batch(A[:20], B[:7], R0)  # more items than one launch takes
    E1 = ctx.tcm_direct_batch(A[:20], B[:7], R0[65530:65540])
    torch.cuda.synchronize()
    assert torch.equal(E[65530:65540], E1)
    E2, E3 = ctx.tcm_direct_batch(A, B, R0[:9]), ctx.tcm_direct(A, B, R0[4])
    torch.cuda.synchronize()
    assert float(E2[4]) == E3


def test_direct_values_that_fixed_point_cannot_hold(ctx):
    """Not finite, overlapping, or outside the radius that was given: as the double loop has it."""
    rng = np.random.default_rng(10)
    A, B = _system(rng, 300, 9.0), _system(rng, 600, 4.0)
    far = np.array([[0.0, 0.0, 60.0]])
    for i, v in ((0, np.nan), (3, np.inf), (3, np.nan)):
        for which in (0, 1):
            X = [A.copy(), B.copy()]
            X[which][17, i] = v
            E = ctx.tcm_direct_batch(*(torch.tensor(x, device="cuda") for x in X), far, cA=np.zeros(3), cB=np.zeros(3))
            assert not np.isfinite(float(E[0])), (which, i, v)
    Ad, Bd = torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda")
    (cA, _), (cB, _) = oracle.center_radius(A), oracle.center_radius(B)
    for R0, rot in ((np.array([1.0, 2.0, 0.5]), None),  # overlapping
                    (far[0], 3.0 * np.eye(3)), (far[0], -np.eye(3))):  # scaled, reflected
        E = ctx.tcm_direct(Ad, Bd, R0, rotB=rot)
        ref, scale = oracle.direct(A, cA, B, cB, R0, rotB=rot, return_abs=True)
        assert abs(E - ref) <= 1e-13 * scale
