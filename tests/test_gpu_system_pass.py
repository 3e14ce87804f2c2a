"""The system pass (centroid, radius, low-degree sums) at the limits of its three kernels: one CTA up
to 8,192 atoms (1,024 double records), a cluster up to 65,536, warp tiles above; float and double records, centre computed or
given.  Centre and radius to double rounding; the mixed path's degrees l <= 2, which come from the
float-float sums (about 2^-44 of their terms), to 1e-11 of the terms' magnitude."""
import numpy as np
import pytest
import torch

import oracle
from paper_0704_1672_gb300 import synth
from tcm_testlib import degree_scales

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0704_1672_gb300 import build
    build.build()
    from paper_0704_1672_gb300 import tcm
    torch.cuda.set_device(0)
    c = tcm.Context(lmax_cap=4)
    yield c
    c.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n", [1, 2, 255, 257, 1024, 1025, 2049, 8191, 8192, 8193, 20000, 65535, 65536, 65537, 70001])
def test_system_pass(ctx, n, dtype):
    from paper_0704_1672_gb300 import tcm
    rng = np.random.default_rng(n)
    S = synth.pack(synth.uniform_ball(rng, n, 25.0) + [100.0, -50.0, 25.0], rng.normal(0.1, 1.0, n))
    t = torch.tensor(S, dtype=dtype, device="cuda")
    S = t.double().cpu().numpy()
    c, a = ctx.tcm_prepare(t)
    c_ref, a_ref = oracle.center_radius(S)
    assert np.allclose(c, c_ref, rtol=0, atol=1e-12 * 100.0)
    assert abs(a - a_ref) <= 1e-12 * max(a_ref, 1.0)
    for centre in (None, np.array([99.0, -49.5, 25.5])):
        m = ctx.tcm_moments(t, 3, precision=tcm.TCM_MIXED, center=centre)
        cc = m.center if centre is None else centre
        ref, sc = oracle.moments(S, cc, 2), degree_scales(S, cc, 2)
        q = tcm.unpack(m.q[:9].cpu(), 2)
        for l in range(3):
            sl = slice(l * l, (l + 1) * (l + 1))
            assert np.max(np.abs(q[sl] - ref[sl])) <= 1e-11 * max(sc[l], 1.0), (l, centre is None)
        d = S[:, :3] - cc
        assert abs(m.radius - np.sqrt((d * d).sum(1).max())) <= 1e-12 * max(m.radius, 1.0)


def test_system_pass_ignores_values_that_are_not_numbers_as_before(ctx):
    """A NaN coordinate does not enter the radius; every size class leaves it finite."""
    for n in (100, 5000, 70000):
        rng = np.random.default_rng(n)
        S = synth.pack(synth.uniform_ball(rng, n, 25.0), rng.normal(size=n))
        S[n // 2, 1] = np.nan
        _, a = ctx.tcm_prepare(torch.tensor(S, dtype=torch.float32, device="cuda"), center=np.zeros(3))
        ok = np.delete(S, n // 2, 0).astype(np.float32).astype(np.float64)
        assert abs(a - np.sqrt((ok[:, :3] ** 2).sum(1).max())) <= 1e-12 * a
