"""The direct sum of systems whose only charges face each other across the gap: 1/r of single pairs, from far
to all but touching, through both forms of the pair loop (csrc/direct.cu), against extended precision.
Double arithmetic rounds B's placed position b' to 2^-53 of its components, and takes six more roundings:
  each 1/r within 2^-53 (|b'| / r + 6) of itself;
  rms over many directions, in units of 2^-53 |b'| / r: sqrt(3/5 x 0.54 / 3) = 0.33 (the mean of the fourth
  powers of a direction's components, of the squared unit in the last place, and of a uniform error), 0.34
  with the other roundings where |b'| / r is about 12; 0.40 leaves three standard errors and a margin.
The rms is taken over narrow gaps, 2^-6 to 2^-4 of the common extent D = R + a_A + a_B, where an error of the
fixed-point form would show first."""
import numpy as np
import pytest
import torch

from paper_0704_1672_gb300 import synth

pytestmark = pytest.mark.gpu


def test_facing_charges():
    from paper_0704_1672_gb300 import build
    build.build()
    from paper_0704_1672_gb300 import tcm
    rng = np.random.default_rng(55)
    worst, near = 0.0, []
    with tcm.Context(lmax_cap=4) as ctx:
        for ax in synth.unit_vectors(rng, 100):
            aA, aB = rng.uniform(10.0, 20.0), rng.uniform(4.0, 20.0)
            A = np.array([[*(aA * ax), 1.0], [*(-aA * ax), 0.0]])
            B = np.array([[*(-aB * ax), 1.0], [*(aB * ax), 0.0]])
            gap = 2.0 * (aA + aB) / (2.0 ** rng.uniform(0.5, 7.0, 200) - 1.0)  # D / gap from 1.4 to 128
            R0 = (aA + aB + gap)[:, None] * ax
            At, Bt = torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda")
            E = ctx.tcm_direct_batch(At, Bt, R0, cA=np.zeros(3), cB=np.zeros(3)).cpu().numpy()
            b = R0.astype(np.longdouble) + B[0, :3].astype(np.longdouble)
            d = b - A[0, :3].astype(np.longdouble)
            r = np.sqrt((d * d).sum(1))
            err = np.abs((E.astype(np.longdouble) * r - 1).astype(np.float64)) * 2.0 ** 53
            placed = (np.sqrt((b * b).sum(1)) / r).astype(np.float64)
            worst = max(worst, float((err / (placed + 6.0)).max()))
            D = 2.0 * (aA + aB) + gap
            at = np.log2(gap / D) + np.log2(D) % 1.0  # log2 of the gap's share, D rounded down to a power of two
            near.append((err / placed)[(at >= -5.0) & (at < -4.0)])
    near = np.concatenate(near)
    rms = float(np.sqrt(np.mean(near ** 2)))
    print(f"worst {worst:.3f} of the bound; rms {rms:.3f} over {len(near)} pairs")
    assert worst <= 1.0 and len(near) > 2000 and rms <= 0.40
