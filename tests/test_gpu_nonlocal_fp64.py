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


# larger contractions run as split products: column tiles of 32 and 16 vectors with remainders,
# projector counts up to the largest, supports of several node chunks, several batches of chunks
# (512 vectors: 8 chunks a batch).  Each size lies past the crossover with the direct kernels.
@pytest.mark.parametrize("npj,nvec,ldx,k", [(32, 16, 16, 0.1), (18, 33, 40, 0.1), (9, 65, 65, -0.2), (18, 65, 66, 0.0),
                                            (18, 512, 512, 0.1), (18, 512, 512, 0.0)])
def test_fp64_nonlocal_split_products(g, npj, nvec, ldx, k):
    chan = {9: (D, P, S), 18: syn.SPD_CHANNELS, 32: CHANNELS[27] + (D,)}[npj]
    big = nvec < 100
    prob = syn.make_problem(ncell=(5, 5, 4) if big else (4, 3, 3), h=(1.0, 1.1, 0.9), p=4 if big else 3,
                            periodic=(1, 1, 0), k=(k, -2 * k, 0.0), natoms=4 if big else 10,
                            rc=2.5 if big else 1.2, seed=npj, channels=chan)
    assert prob.atoms[0].npj == npj
    X = syn.random_block(prob.nnodes, nvec, 3)
    X *= np.logspace(-8, 8, nvec)                    # columns of very different size
    ref = fe.Discretisation(prob).apply_h(X)
    Xd = torch.zeros((prob.nnodes, 2, ldx), dtype=torch.complex128, device="cuda")
    Xd[:, :, :nvec] = torch.from_numpy(X).cuda()
    ctx = g.Context(0)
    ctx.set_problem(prob)
    Y = torch.empty_like(Xd)
    ctx.apply_h(Xd, Y, nvec=nvec)
    ctx.sync_status()
    got = Y[:, :, :nvec].cpu().numpy()
    err = np.linalg.norm(got - ref, axis=(0, 1))
    assert (err <= 1e-12 * np.linalg.norm(ref, axis=(0, 1))).all()
    if not big:
        return
    # a NaN and an infinity reach their own columns only
    Xd[prob.nnodes // 2, 0, 1] = float("nan")
    Xd[prob.nnodes // 2, 1, 4] = float("inf")
    ctx.apply_h(Xd, Y, nvec=nvec)
    ctx.sync_status()
    again = Y[:, :, :nvec].cpu().numpy()
    assert set(np.flatnonzero(~np.isfinite(again).all(axis=(0, 1)))) == {1, 4}
    rest = [v for v in range(nvec) if v not in (1, 4)]
    again = again[:, :, rest]
    assert np.linalg.norm(again - ref[:, :, rest]) <= 1e-12 * np.linalg.norm(ref[:, :, rest])
