"""The radius where the float filter cannot tell the atoms apart: every atom of a shell within the
filter's margin, so that a lane holds several candidates, and values beyond the float range of the
square.  The radius is the exact double maximum: 1e-12 relative, as elsewhere."""
import numpy as np
import pytest
import torch

from paper_0704_1672_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 300, 513, 9000, 70001])
@pytest.mark.parametrize("scale", [1.0, 1e25])
@pytest.mark.parametrize("spread", [0.0, 1e-6, 1e-4])
def test_radius_of_a_shell(n, scale, spread):
    from paper_0704_1672_gb300 import build
    build.build()
    from paper_0704_1672_gb300 import tcm
    rng = np.random.default_rng(n)
    v = rng.normal(size=(n, 3))
    x = v / np.linalg.norm(v, axis=1)[:, None] * 30.0 * (1.0 + spread * rng.uniform(-1.0, 1.0, (n, 1)))
    t = torch.tensor(synth.pack(x * scale, rng.normal(size=n)), dtype=torch.float32, device="cuda")
    X = t.double().cpu().numpy()[:, :3]
    with tcm.Context(lmax_cap=4) as ctx:
        _, a = ctx.tcm_prepare(t, center=np.zeros(3))
        m = ctx.tcm_moments(t, 2, precision=tcm.TCM_MIXED, center=np.zeros(3)) if scale == 1.0 else None
    ref = np.sqrt((X * X).sum(1).max())
    assert abs(a - ref) <= 1e-12 * ref
    assert m is None or abs(m.radius - ref) <= 1e-12 * ref


def test_radius_of_an_atom_at_infinity():
    from paper_0704_1672_gb300 import tcm
    for n in (100, 9000, 70001):
        S = synth.pack(synth.uniform_ball(np.random.default_rng(n), n, 25.0), np.ones(n))
        S[n // 3, 2] = np.inf
        with tcm.Context(lmax_cap=4) as ctx:
            _, a = ctx.tcm_prepare(torch.tensor(S, dtype=torch.float32, device="cuda"), center=np.zeros(3))
        assert np.isinf(a)
