"""FP32 cell apply at the orders and shapes where its thread groups, plane ownership and
tables change: p = 3, 4, 5 (group sizes) and p = 6 (planes owned by warps), unequal cell
edges (the z kinetic operator carries the x and y edges), Dirichlet faces in every
direction, ragged vector chunks and several systems in one launch.

Tolerances as test_gpu_batch.py: H.X relative Frobenius 1e-5, degree-3 filter 2e-5."""
import numpy as np
import pytest

import synthetic as syn
from oracle import chfsi as oc
from oracle import fe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import __graft_entry__ as ge
    ge.build()
    import paper_2410_02754_gb300 as pkg
    return pkg


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


CASES = [((3, 2, 1), 3, (1, 0, 1), (0.1, 0.0, -0.2), 3), ((1, 2, 3), 4, (0, 1, 0), (0.0, 0.0, 0.0), 9),
         ((2, 1, 2), 5, (1, 1, 0), (0.0, 0.2, 0.1), 5), ((2, 3, 1), 6, (0, 0, 0), (0.05, 0.1, 0.2), 6)]


@pytest.mark.parametrize("var", [0, 1, 2, 4])
@pytest.mark.parametrize("case", CASES, ids=lambda c: f"p{c[1]}")
def test_cell_groups(g, var, case):
    ncell, p, per, k, nvec = case
    prob = syn.make_problem(ncell=ncell, h=(0.9, 1.3, 1.1), p=p, periodic=per, k=k, natoms=1, rc=0.8,
                            seed=31)
    d = fe.Discretisation(prob)
    X = syn.random_block(d.mesh.nnodes, nvec, 8)
    c = g.Context(0)
    c.set_problem(prob)
    c.set_precision(1)
    c.set_cell_variant(var)
    Xd = torch.from_numpy(X).to(torch.complex64).cuda()
    Yd = torch.empty_like(Xd)
    c.apply_h(Xd, Yd)
    c.sync_status()
    assert rel(Yd.cpu().numpy(), d.apply_h(X)) < 1e-5
    bounds = (1.0, 90.0, -2.0)
    c.filter(Xd, 3, *bounds)
    c.sync_status()
    assert rel(Xd.cpu().numpy().astype(np.complex128), oc.cheb_filter(d.apply_htilde, X, 3, *bounds)) < 2e-5
    c.close()


@pytest.mark.parametrize("p", [3, 4, 5, 6, 7])
def test_local_apply_keeps_fp32_accuracy(g, p):
    """FP32 against FP64 H.X of a uniform random block, no projectors, k = 0.  The same operator as
    separate kinetic and potential passes, every table rounded to FP32 once and every operation
    once, is off by 0.86e-7 to 1.04e-7 for p = 3 .. 7 (emulated): no more than 1.05e-7."""
    prob = syn.make_problem(ncell=(4, 3, 3), h=(1.0, 1.0, 1.0), p=p, seed=2)
    c = g.Context(0)
    c.set_problem(prob)
    X = torch.rand((prob.nnodes, 2, 8, 2), device="cuda",
                   generator=torch.Generator("cuda").manual_seed(p)) * 2 - 1
    X = torch.view_as_complex(X)
    ref = torch.empty(X.shape, dtype=torch.complex128, device="cuda")
    c.apply_h(X.to(torch.complex128), ref)
    c.set_precision(1)
    Y = torch.empty_like(X)
    for var in (0, 2, 4):
        c.set_cell_variant(var)
        c.apply_h(X, Y)
        assert float((Y - ref).norm() / ref.norm()) < 1.05e-7
    c.close()


@pytest.mark.parametrize("p,ncell,nvec", [(2, (12, 10, 10), 17), (5, (8, 7, 6), 9), (6, (7, 6, 6), 11), (7, (7, 6, 5), 13)])
def test_groups_take_many_items(g, p, ncell, nvec):
    """More work items than the GPU has groups, so that every group reuses its item slots: H.X of both
    precisions and the fused FP32 recurrence, with a ragged last vector chunk and Dirichlet faces."""
    prob = syn.make_problem(ncell=ncell, h=(0.9, 1.0, 1.1), p=p, periodic=(1, 0, 1), k=(0.1, 0.0, -0.1), seed=p)
    d = fe.Discretisation(prob)
    X = syn.random_block(d.mesh.nnodes, nvec, 4)
    want = d.apply_h(X)
    bounds = (1.0, 300.0, -3.0)
    c = g.Context(0)
    c.set_problem(prob)
    X64 = torch.from_numpy(X).cuda()
    Y64 = torch.empty_like(X64)
    c.apply_h(X64, Y64)
    assert rel(Y64.cpu().numpy(), want) < 1e-12
    F64 = X64.clone()
    c.filter(F64, 3, *bounds)
    c.set_precision(1)
    X32 = X64.to(torch.complex64)
    for var in (0, 2, 4):
        c.set_cell_variant(var)
        Y = torch.empty_like(X32)
        c.apply_h(X32, Y)
        c.sync_status()
        assert rel(Y.cpu().numpy(), want) < 1e-5
        F = X32.clone()
        c.filter(F, 3, *bounds)
        c.sync_status()
        assert rel(F.cpu().numpy(), F64.cpu().numpy()) < 2e-5
    c.close()
