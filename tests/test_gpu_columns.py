"""The float moment pass by columns (few tiles) and by chunks (many) must give the same bits: an item
alone takes the first, in a batch of many distinct moment sets the second.  Sizes around the row, batch
and tile limits (32, 128 and 2,048 atoms), both chunk budgets, float and double records."""
import numpy as np
import pytest
import torch

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


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("kmax", [160, 96])
def test_columns_give_the_chunk_kernels_bits(tcm, kmax, dtype):
    rng = np.random.default_rng(kmax)
    sizes = [1, 31, 33, 127, 129, 2047, 2049, 4500]
    systems = [synth.pack(synth.uniform_ball(rng, n, 9.0) + [5.0, -2.0, 1.0], rng.normal(size=n)) for n in sizes]
    T = [(torch.tensor(S, dtype=dtype, device="cuda"), None, None) for S in systems]
    with tcm.Context(lmax_cap=24) as ctx:
        for L in range(25):
            ctx.tcm_ctx_set_chunking_l(L, kmax)
        for L in range(25):
            k = 200  # at least 200 moment sets: more tiles than SMs
            a, b = np.arange(k) % len(sizes), (np.arange(k) // 2) % len(sizes)
            R0, rot = synth.unit_vectors(rng, k) * 40.0, synth.random_rotations(rng, k)
            E, _ = ctx.tcm_energy_batch(T, a, b, np.full(k, L), R0, rotB=rot)
            for i in range(0, 2 * len(sizes), 2):
                Ei, _ = ctx.tcm_energy_batch(T, a[i:i + 1], b[i:i + 1], [L], R0[i:i + 1], rotB=rot[i:i + 1])
                torch.cuda.synchronize()
                assert float(Ei[0]) == float(E[i]), (L, i, float(Ei[0]) - float(E[i]))
