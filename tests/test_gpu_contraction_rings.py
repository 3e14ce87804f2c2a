"""Two coaxial rings of n alternating unit charges stacked along R0: their lowest moment is l = m = n/2, so
at Lmax = l one (l1, l2) block is the whole energy, carried by its highest order.  With
Q_ll = n r^l sqrt(C(2l, l)) / 2^l about the axis, Eq. (Formula) is
    E = K cos(l t),  K = 2 n^2 (r_A r_B)^l C(2l, l) / 4^l / R^(2l+1),
t the angle between the rings: the force on B is (2l+1) E / R along R0, the torque on B K l sin(l t) about
R0 and that on A its opposite.  In double, for every way B's moments reach the contraction, at the 1e-12
bar; the rounding of the rings' coordinates moves these values by about l 2e-16 of themselves.  (The
oracle sums over lab-frame harmonics, which cancel for axes off z; the closed form does not.)"""
import math

import numpy as np
import pytest
import torch

from tcm_testlib import TOL_FP64

pytestmark = pytest.mark.gpu

RA, RB, R = 10.0, 8.0, 18.5  # ring radii and separation: closer rings, so that rounding leaves no lower moment of note
AXES = {"z": np.array([0.0, 0.0, 1.0]), "x": np.array([1.0, 0.0, 0.0]), "generic": np.array([12.0, -16.0, 15.0]) / 25.0}


@pytest.fixture(scope="module")
def tcm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0704_1672_gb300 import build
    build.build()
    from paper_0704_1672_gb300 import tcm as t
    torch.cuda.set_device(0)
    return t


def ring(n, r, t, u, v):
    phi = 2.0 * np.pi * np.arange(n) / n + t
    x = r * (np.cos(phi)[:, None] * u + np.sin(phi)[:, None] * v)
    return np.concatenate([x, np.where(np.arange(n) % 2 == 0, 1.0, -1.0)[:, None]], axis=1)


def closed_form(n, rb, t):
    """E, the force along R0 and the torque on B about it."""
    l = n // 2
    K = 2.0 * n * n * (RA * rb) ** l * math.comb(2 * l, l) / 4.0 ** l / R ** (2 * l + 1)
    return K * math.cos(l * t), (2 * l + 1) * K * math.cos(l * t) / R, K * l * math.sin(l * t)


def axis_rotation(ax, angle):
    k = np.array([[0.0, -ax[2], ax[1]], [ax[2], 0.0, -ax[0]], [-ax[1], ax[0], 0.0]])
    return np.eye(3) + math.sin(angle) * k + (1.0 - math.cos(angle)) * (k @ k)


@pytest.mark.parametrize("axis", list(AXES))
@pytest.mark.parametrize("n", [4, 8, 12, 16, 24, 32, 40, 48])
def test_coaxial_rings_fp64(tcm, n, axis):
    ax, L = AXES[axis], n // 2
    h = np.eye(3)[int(np.argmin(np.abs(ax)))]
    u = np.cross(ax, h)
    u /= np.linalg.norm(u)
    v = np.cross(ax, u)
    t0, t1, grow = 0.3 / n, 0.1 / n, 1.0 + 2.0 ** -20
    At, Bt = (torch.tensor(x, device="cuda") for x in (ring(n, RA, 0.0, u, v), ring(n, RB, t0, u, v)))
    turn = axis_rotation(ax, t1)
    c, R0 = np.zeros(3), ax * R
    with tcm.Context(lmax_cap=24) as ctx:
        mA = ctx.tcm_moments(At, L, precision=tcm.TCM_FP64, center=c)
        mB = ctx.tcm_moments(Bt, L, precision=tcm.TCM_FP64, center=c)
        E0 = closed_form(n, RB, t0)[0]
        assert abs(ctx.tcm_energy(mA, mB, R0, L) - E0) <= TOL_FP64 * abs(E0)
        cached = [tcm.make_system(At, c, mA.radius, moments=mA), tcm.make_system(Bt, c, mB.radius, moments=mB)]
        plain = [(At, c, None), (Bt, c, None)]
        for systems, rot, rb, t in ((plain, None, RB, t0),                # both sides in the lab frame
                                    (plain, turn, RB, t0 + t1),           # B's lab-frame set rotated
                                    (plain, turn * grow, RB * grow, t0 + t1),  # no rotation: B's atoms are moved
                                    (cached, turn, RB, t0 + t1)):         # B's moment cache rotated
            ctx.tcm_ctx_set_rotate_cached(systems is cached)
            rots = None if rot is None else rot[None]
            E, G, st = ctx.tcm_gradients_batch(systems, [0], [1], [L], R0[None], rotB=rots, precision=tcm.TCM_FP64)
            E2, _ = ctx.tcm_energy_batch(systems, [0], [1], [L], R0[None], rotB=rots, precision=tcm.TCM_FP64)
            torch.cuda.synchronize()
            assert int(st[0]) == 0 and torch.equal(E, E2)
            E, G = float(E[0]), G[0].cpu().numpy()
            e, f, tau = closed_form(n, rb, t)
            assert abs(E - e) <= TOL_FP64 * abs(e), (E, e)
            assert np.linalg.norm(G[:3] - f * ax) <= TOL_FP64 * abs(f)
            assert np.linalg.norm(G[3:6] + tau * ax) <= TOL_FP64 * L * abs(e)
            assert np.linalg.norm(G[6:] - tau * ax) <= TOL_FP64 * L * abs(e)
