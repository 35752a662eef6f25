"""The eigensolver and the Lanczos process at the edges of their blocks: matrices of 1 to 17
columns (odd orders, pair blocks of 8, a pair without partner) and 1 to 20 Lanczos steps (basis
groups of 8 with remainders), in the default and the fixed-order mode.

Tolerances: Ritz values 1e-11 of the largest (FP64, as test_gpu_split_products.py); Lanczos bounds
1e-9 relative, as test_gpu_parity.py::test_lanczos_bounds_match_oracle compares them."""
import numpy as np
import pytest

import synthetic as syn
from oracle import chfsi as oc
from oracle import fe

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    import __graft_entry__ as ge
    ge.build()
    import paper_2410_02754_gb300 as g
    prob = syn.make_problem(ncell=(2, 2, 2), h=(1.0, 1.1, 1.2), p=3, k=(0.1, 0.0, -0.1), natoms=1, rc=1.0,
                            seed=8)
    ctx = g.Context(0)
    ctx.set_problem(prob)
    return ctx, prob, fe.Discretisation(prob)


@pytest.mark.parametrize("n", [1, 2, 3, 7, 15, 16, 17])
def test_ritz_values_of_small_blocks(setup, n):
    ctx, prob, d = setup
    X = torch.from_numpy(syn.random_block(prob.nnodes, n, 40 + n)).cuda()
    ctx.cholgs(X)
    x = X.cpu().numpy()
    ref = np.linalg.eigvalsh(x.reshape(-1, n).conj().T @ d.apply_h(x).reshape(-1, n))
    ritz = ctx.rayleigh_ritz(X)
    assert np.abs(ritz - ref).max() <= 1e-11 * np.abs(ref).max()
    y = X.cpu().numpy()
    Hp = y.reshape(-1, n).conj().T @ d.apply_h(y).reshape(-1, n)
    assert np.abs(Hp - np.diag(ritz)).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("det", [False, True])
@pytest.mark.parametrize("steps", [1, 2, 8, 9, 17, 20])
def test_lanczos_steps(setup, steps, det):
    ctx, prob, d = setup
    v0 = syn.random_start(prob.nnodes, 3)
    ref = oc.lanczos_bounds(d.apply_htilde, d.md, v0, steps)
    ctx.set_deterministic(det)
    got = ctx.lanczos_bounds(torch.from_numpy(v0).cuda(), steps)
    ctx.set_deterministic(False)
    assert np.abs(np.subtract(got, ref)).max() < 1e-9 * abs(ref[1])
