"""FP64 projection and atom-major expansion at the edges of their tiles: column tiles of 2 to
32 with remainders, projector counts at and between the compiled ones, supports that share
nodes, a padded leading dimension, and the fixed-order (deterministic) sums.

Tolerance: FP64 H.X against the oracle, relative Frobenius 1e-12 (as test_gpu_parity.py)."""
import numpy as np
import pytest

import synthetic as syn
from oracle import fe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

S, P, D = (0.5, 0), (0.6, 1), (0.5, 2)
CHANNELS = {1: (S,), 4: (S, P), 8: (D, P), 18: syn.SPD_CHANNELS, 27: syn.SPD_CHANNELS + (D, P, S)}


@pytest.fixture(scope="module")
def g():
    import __graft_entry__ as ge
    ge.build()
    import paper_2410_02754_gb300 as pkg
    return pkg


@pytest.mark.parametrize("npj,nvec,ldx", [(1, 1, 1), (4, 2, 2), (8, 3, 5), (18, 1, 1), (18, 8, 8),
                                          (18, 16, 16), (18, 17, 20), (27, 33, 33)])
def test_fp64_nonlocal_tiles(g, npj, nvec, ldx):
    prob = syn.make_problem(ncell=(4, 3, 3), h=(1.0, 1.1, 0.9), p=3, periodic=(1, 1, 0),
                            k=(0.1, -0.2, 0.0), natoms=3, rc=1.6, seed=npj, channels=CHANNELS[npj])
    assert prob.atoms[0].npj == npj
    X = syn.random_block(prob.nnodes, nvec, 3)
    ref = fe.Discretisation(prob).apply_h(X)
    Xd = torch.zeros((prob.nnodes, 2, ldx), dtype=torch.complex128, device="cuda")
    Xd[:, :, :nvec] = torch.from_numpy(X).cuda()
    ctx = g.Context(0)
    ctx.set_problem(prob)
    for det in (False, True):
        ctx.set_deterministic(det)
        Y = torch.empty_like(Xd)
        ctx.apply_h(Xd, Y, nvec=nvec)
        ctx.sync_status()
        got = Y[:, :, :nvec].cpu().numpy()
        assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
