"""FP64 cell apply at the edges of its pairing: every order, unequal cell edges, Dirichlet
faces, one vector (pairs of cells), odd products of cells and vectors (an absent second
half of the last pair), a padded leading dimension, and the per-cell (deterministic) mode.

Tolerance: FP64 H.X against the oracle, relative Frobenius 1e-12 (as test_gpu_parity.py)."""
import numpy as np
import pytest

import synthetic as syn
from oracle import fe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import __graft_entry__ as ge
    ge.build()
    import paper_2410_02754_gb300 as pkg
    return pkg


@pytest.mark.parametrize("p,ncell,per,nvec,ldx", [
    (2, (3, 1, 1), (1, 0, 1), 1, 1), (3, (1, 3, 5), (1, 1, 1), 1, 2), (4, (3, 2, 2), (0, 0, 0), 5, 5),
    (5, (2, 2, 1), (1, 1, 0), 3, 4), (6, (3, 1, 3), (1, 0, 1), 7, 7), (6, (1, 1, 1), (0, 1, 1), 2, 2),
    (7, (1, 2, 1), (1, 1, 1), 3, 3)])
def test_fp64_cell_pairs(g, p, ncell, per, nvec, ldx):
    k = (0.1, 0.0, -0.2) if p % 2 else (0.0, 0.0, 0.0)
    prob = syn.make_problem(ncell=ncell, h=(0.9, 1.3, 1.1), p=p, periodic=per, k=k, seed=p)
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


@pytest.mark.parametrize("p", [4, 7])
def test_fp64_items_of_one_and_two(g, p):
    """The numbers of (cell, vector)s at which the items of the cell apply change from one to two and
    back: around 1, 2 and 3 for every SM, odd and even."""
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    for n in (1, sm, sm + 1, 2 * sm, 2 * sm + 1, 3 * sm, 3 * sm + 1):
        prob = syn.make_problem(ncell=(n, 1, 1), h=(0.9, 1.3, 1.1), p=p, periodic=(1, 1, 0),
                                k=(0.1, 0.0, 0.0) if n % 2 else (0.0, 0.0, 0.0), seed=n)
        X = syn.random_block(prob.nnodes, 1, 3)
        ref = fe.Discretisation(prob).apply_h(X)
        ctx = g.Context(0)
        ctx.set_problem(prob)
        Xd = torch.from_numpy(X).cuda()
        Y = torch.empty_like(Xd)
        ctx.apply_h(Xd, Y)
        assert np.linalg.norm(Y.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
        ctx.close()
