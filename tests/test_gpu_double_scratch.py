"""Scratch of the double path's moment pass: a row of partial sums holds its degree's components, and a batch
whose rows pass 1 GiB runs in several passes over the same rows.  Every item has the bits of a call
of its own, whatever pass it falls into and whatever degrees stand beside it."""
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


def _batch(tcm, n, k, L):
    """k pairs of one atom set about centres of their own (2 k moment sets), |R0| = 60, degrees L."""
    rng = np.random.default_rng(n + k)
    X = torch.tensor(synth.pack(synth.uniform_ball(rng, n, 20.0), rng.normal(size=n)), device="cuda")
    systems = [tcm.make_system(X, center=c, radius=25.0) for c in rng.normal(size=(2 * k, 3))]
    R0 = synth.unit_vectors(rng, k) * 60.0
    return X, systems, np.arange(k), np.arange(k, 2 * k), np.asarray(L), R0


def _check(tcm, ctx, batch, items):
    _, systems, a, b, L, R0 = batch
    E, st = ctx.tcm_energy_batch(systems, a, b, L, R0, precision=tcm.TCM_FP64)
    torch.cuda.synchronize()
    assert bool(torch.all(st == 0))
    for k in items:
        E1, _ = ctx.tcm_energy_batch([systems[a[k]], systems[b[k]]], [0], [1], [L[k]], R0[k:k + 1], precision=tcm.TCM_FP64)
        assert float(E1[0]) == float(E[k]), k
    return E


@pytest.mark.parametrize("mode", [0, 2])  # launched, captured
def test_batches_of_several_passes(tcm, mode):
    k = 2200  # 4,400 sets of 2,000 atoms, 63 rows of up to 625 doubles: 1.2 GB, two passes
    L = np.where(np.arange(k) % 8 == 7, 23, 24)
    batch = _batch(tcm, 2000, k, L)
    with tcm.Context(lmax_cap=24) as ctx:
        ctx.tcm_ctx_set_graphs(mode)
        # pass 1 ends after 2^27 / (63 x 625) sets, near 3,409 + the shorter rows' gain
        items = [0, 1, 7, 1150, 1200, 1207, 1208, 1250, 1300, k - 1]
        E = _check(tcm, ctx, batch, items)
        assert torch.equal(E, _check(tcm, ctx, batch, []))


def test_rows_of_small_degrees(tcm):
    """20,000 sets of 2,000 atoms at degree 4 need 250 MB of rows."""
    k = 10000
    batch = _batch(tcm, 2000, k, np.full(k, 4))
    torch.cuda.synchronize()
    with tcm.Context(lmax_cap=24) as ctx:
        free = torch.cuda.mem_get_info()[0]
        _check(tcm, ctx, batch, [0, 1, 5000, k - 1])
        assert free - torch.cuda.mem_get_info()[0] < 768 << 20
        small = _batch(tcm, 300, 40, np.arange(40) % 25)  # every degree in one call
        _check(tcm, ctx, small, range(40))
