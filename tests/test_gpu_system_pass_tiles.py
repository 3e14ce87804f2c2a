"""Systems above 65,536 atoms with a given centre: the radius and low-degree sums are then the first pass
over the atoms, behind the kernel that writes its tiles or descriptors (the fixed scratch's preparation,
a long tile list), and must not read them ahead of it.  Calls on two systems in turn, so that a descriptor
of the call before would show.  Radius to double rounding, degrees l <= 2 to 1e-11 of their terms
(float-float sums, about 2^-44), the others as the parity tests have them."""
import numpy as np
import pytest
import torch

import oracle
from paper_0704_1672_gb300 import synth
from tcm_testlib import TOL_MIX_MOM, degree_scales, moment_error, oracle_moments_threaded

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


def _systems(sizes):
    out = []
    for n in sizes:
        rng = np.random.default_rng(n)
        S = synth.pack(synth.uniform_ball(rng, n, 30.0), rng.normal(0.05, 1.0, n)).astype(np.float32)
        out.append((torch.tensor(S, device="cuda"), S.astype(np.float64), rng.normal(size=3)))
    return out


def _check_low(q, radius, S, c, tcm):
    ref, sc = oracle.moments(S, c, 2), degree_scales(S, c, 2)
    got = tcm.unpack(q[:9].cpu(), 2)
    for l in range(3):
        sl = slice(l * l, (l + 1) * (l + 1))
        assert np.max(np.abs(got[sl] - ref[sl])) <= 1e-11 * max(sc[l], 1.0), l
    d = S[:, :3] - c
    a = np.sqrt((d * d).sum(1).max())
    assert abs(radius - a) <= 1e-12 * a


@pytest.mark.parametrize("sizes", [(65537, 70001), (200000, 65600)])
def test_fixed_scratch_with_a_given_centre(tcm, sizes):
    systems, L = _systems(sizes), 6
    refs = [oracle_moments_threaded(S, c, L) for _, S, c in systems]
    for _ in range(10):
        outs = []
        for X, _, c in systems:
            q = torch.empty((L + 1) ** 2, dtype=torch.float64, device="cuda")
            g = torch.empty(4, dtype=torch.float64, device="cuda")
            tcm.tcm_moments_noalloc(X, L, tcm.TCM_MIXED, center=c, out=q, center_radius_out=g)
            outs.append((q, g))
        torch.cuda.synchronize()
        for (q, g), (_, S, c), ref in zip(outs, systems, refs):
            _check_low(q, float(g[3]), S, c, tcm)
            assert moment_error(tcm.unpack(q), ref, degree_scales(S, c, L)) < TOL_MIX_MOM


def test_long_tile_list_with_a_given_centre(tcm):
    systems = _systems((1000000, 900001))  # 2,445 and 2,200 moment tiles and 977 and 879 of the system pass
    with tcm.Context(lmax_cap=24) as ctx:
        for _ in range(5):
            for X, S, c in systems:
                m = ctx.tcm_moments(X, 24, precision=tcm.TCM_MIXED, center=c)
                _check_low(m.q, m.radius, S, c, tcm)
