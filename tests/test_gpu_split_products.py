"""CholGS and Rayleigh-Ritz through the split tensor-core products (16 columns and more), at
the edges of their tiles (64- and 128-wide, padded columns, the largest block), with a padded
leading dimension, columns and rows of very different size, and blocks that are not finite or
not of full rank.

FP64 blocks: X^H M X = I and the span to 1e-12 (the FP64 rounding of test_gpu_parity.py).  FP32
blocks: one rounding to FP32 per entry, so the rotated columns agree with the FP64 result to
2^-23 of a column (a rounding error is at most 2^-24 of an entry, and the input is exact)."""
import numpy as np
import pytest

import synthetic as syn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import __graft_entry__ as ge
    ge.build()
    import paper_2410_02754_gb300 as pkg
    return pkg


def block(M, n, seed):
    """Columns from 1 to 1e-3, rows falling off by 1e-1.5, neighbouring columns overlapping."""
    X = syn.random_block(M, n, seed)
    X[:, :, 1:] += 0.4 * X[:, :, :-1]
    return X * np.logspace(0, -1.5, M)[:, None, None] * np.logspace(0, -3, n)


def context(g, prec, ncell=(3, 3, 3), p=5):
    prob = syn.make_problem(ncell=ncell, h=(1.0, 1.1, 0.9), p=p, k=(0.1, 0.0, 0.0), natoms=1, rc=1.0, seed=4)
    ctx = g.Context(0)
    ctx.set_problem(prob)
    ctx.set_precision(prec)
    return ctx, prob


def device(X, prec, ldx):
    out = torch.zeros(X.shape[:2] + (ldx,), dtype=torch.complex64 if prec else torch.complex128, device="cuda")
    out[:, :, :X.shape[2]] = torch.from_numpy(X).to(out.dtype).cuda()
    return out


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,ldx", [(15, 15), (16, 17), (33, 33), (64, 64), (65, 70), (129, 129), (512, 512)])
def test_cholgs_tiles(g, prec, n, ldx):
    ctx, prob = context(g, prec)
    M = prob.nnodes
    Xd = device(block(M, n, 3), prec, ldx)
    X = Xd[:, :, :n].cpu().numpy().astype(np.complex128).reshape(2 * M, n)   # the exact input
    md = np.repeat(ctx.mass(), 2)[:, None]
    L = np.linalg.cholesky(X.conj().T @ (md * X))
    ref = np.linalg.solve(L.conj(), X.T).T          # X L^-H
    ctx.cholgs(Xd, nvec=n)
    Y = Xd[:, :, :n].cpu().numpy().astype(np.complex128).reshape(2 * M, n)
    if prec == 0:
        G = Y.conj().T @ (md * Y)
        assert np.abs(G - np.eye(n)).max() < 1e-12
    err = np.linalg.norm(Y - ref, axis=0) / np.linalg.norm(ref, axis=0)
    assert err.max() < (1e-12 if prec == 0 else 2.0 ** -23)
    if ldx > n:
        assert not Xd[:, :, n:].any()
    ctx.close()


@pytest.mark.parametrize("prec,n", [(0, 16), (0, 65), (1, 65), (1, 130)])
def test_cholgs_columns_of_any_size(g, prec, n):
    """Column sizes over the type's range: CholGS does not depend on a column's size, so the same
    block with its columns at 1, 2^-66, 2^-116 and 2^-332 (FP32: 2^-98, about 1e-30) of themselves
    gives the same orthonormal block."""
    ctx, prob = context(g, prec)
    M = prob.nnodes
    X = device(block(M, n, 3), prec, n).cpu().numpy().astype(np.complex128)
    md = np.repeat(ctx.mass(), 2)[:, None]
    f = X.reshape(2 * M, n)
    L = np.linalg.cholesky(f.conj().T @ (md * f))
    ref = np.linalg.solve(L.conj(), f.T).T
    shift = np.array([0, -66, -116, -332] if prec == 0 else [0, -66, -98])
    Xd = device(X * np.exp2(shift[np.arange(n) * 7 % len(shift)].astype(float)), prec, n)
    ctx.cholgs(Xd)
    Y = Xd.cpu().numpy().astype(np.complex128).reshape(2 * M, n)
    if prec == 0:
        assert np.abs(Y.conj().T @ (md * Y) - np.eye(n)).max() < 1e-12
    err = np.linalg.norm(Y - ref, axis=0) / np.linalg.norm(ref, axis=0)
    assert err.max() < (1e-12 if prec == 0 else 2.0 ** -23)
    ctx.close()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [16, 63, 130])
def test_rayleigh_ritz_tiles(g, prec, n):
    from oracle import fe
    ctx, prob = context(g, prec, (2, 2, 3), 4)
    d = fe.Discretisation(prob)
    Xd = device(block(prob.nnodes, n, 5), prec, n)
    ctx.cholgs(Xd)
    X = Xd.cpu().numpy().astype(np.complex128)
    flat = X.reshape(-1, n)
    ref = np.linalg.eigvalsh(flat.conj().T @ d.apply_h(X).reshape(-1, n))
    ritz = ctx.rayleigh_ritz(Xd)
    assert np.abs(ritz - ref).max() < 1e-11 * np.abs(ref).max()
    Y = Xd.cpu().numpy().astype(np.complex128)
    Hp = Y.reshape(-1, n).conj().T @ d.apply_h(Y).reshape(-1, n)
    off = Hp - np.diag(np.diag(Hp))
    assert np.abs(off).max() < (1e-11 if prec == 0 else 1e-5) * np.abs(ref).max()
    ctx.close()


def test_gram_of_peaked_columns(g):
    """Columns that peak in one of 746,000 rows: an FP64 sum of K terms in 64 parts is off by about
    sqrt(K / 64) 2^-53 of its value, and the block of CholGS is orthonormal to that."""
    ctx, prob = context(g, 0, (12, 12, 12), 6)
    M, n = prob.nnodes, 16
    Xd = torch.rand((M, 2, n, 2), dtype=torch.float64, device="cuda",
                    generator=torch.Generator("cuda").manual_seed(1)) * 2 - 1
    Xd = torch.view_as_complex(Xd)
    Xd[M // 3, 0] *= 1000.0
    ctx.cholgs(Xd)
    Y = Xd.reshape(2 * M, n)
    md = torch.from_numpy(np.repeat(ctx.mass(), 2)).cuda()[:, None]
    G = sum(y.mH @ (m * y) for y, m in zip(Y.chunk(512), md.chunk(512)))
    off = float((G - torch.eye(n, device="cuda")).abs().max())
    assert off < (2 * M / 64) ** 0.5 * 2.0 ** -53
    ctx.close()


def localised(prob, n):
    """Columns peaked on one interior node of a cell each, a weak random tail everywhere."""
    nx, ny, nz = prob.ncell
    p, M = prob.p, prob.nnodes
    cell = np.arange(n)
    g = [c * p + 1 for c in (cell % nx, cell // nx % ny, cell // (nx * ny))]
    X = 1e-4 * syn.random_block(M, n, 9)
    X[(g[2] * ny * p + g[1]) * nx * p + g[0], 0, cell] += 1.0
    return X


@pytest.mark.parametrize("n,local", [(32, False), (256, False), (128, True), (512, True)])
def test_ritz_rotation_of_a_converged_fp32_block(g, n, local):
    """An FP32 block that is rotated close to the identity is rounded to FP32 once: what X Q leaves
    over in the rotated block (least squares for Q) is at most 2^-24 of each column, however
    delocalised or localised the columns are."""
    ncell, p = ((8, 8, 8), 3) if local else ((3, 3, 3), 5)
    prob = syn.make_problem(ncell=ncell, h=(1.0, 1.1, 0.9), p=p, seed=4)
    if local:   # one potential per cell: the localised columns are close to eigenvectors
        prob = prob.with_(veff=prob.veff + 0.5 * np.arange(512.0)[:, None])
    ctx = g.Context(0)
    ctx.set_problem(prob)
    ctx.set_precision(1)
    Xd = device(localised(prob, n) if local else block(prob.nnodes, n, 5), 1, n)
    ctx.cholgs(Xd)
    ctx.rayleigh_ritz(Xd)
    # Ritz vectors turned a little, as a filter leaves them: the next Q is close to the identity
    K = 1e-3 / n ** 0.5 * torch.randn((n, n), dtype=torch.complex128, device="cuda",
                                      generator=torch.Generator("cuda").manual_seed(n))
    Xd += (Xd.to(torch.complex128) @ (K - K.mH)).to(Xd.dtype)
    ctx.cholgs(Xd)
    X = Xd.to(torch.complex128).reshape(-1, n)
    ctx.rayleigh_ritz(Xd)
    Y = Xd.to(torch.complex128).reshape(-1, n)
    Q = torch.linalg.solve(X.mH @ X, X.mH @ Y)
    left = torch.linalg.vector_norm(Y - X @ Q, dim=0) / torch.linalg.vector_norm(Y, dim=0)
    assert float(left.max()) < 2.0 ** -24
    ctx.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_cholgs_refuses_what_it_refused(g, prec):
    ctx, prob = context(g, prec, (2, 2, 2), 3)
    for bad in (np.inf, np.nan, 0.0):
        X = syn.random_block(prob.nnodes, 20, 6)
        if bad == 0.0:
            X[:, :, 7] = 0.0
        else:
            X[11, 1, 7] = bad
        Xd = device(X, prec, 20)
        keep = Xd.clone()
        with pytest.raises(g.GbcError) as e:
            ctx.cholgs(Xd)
        assert e.value.status == 5                       # GBC_ENOTPD, the block unchanged
        assert torch.equal(torch.view_as_real(Xd).nan_to_num(), torch.view_as_real(keep).nan_to_num())
    ctx.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_no_memory_for_the_digits(g, prec):
    """With too little device memory for the digits, CholGS and Rayleigh-Ritz run the direct kernels
    (which need one more block), and the digits kept from an earlier call make room for other work."""
    ctx, prob = context(g, prec, (6, 6, 6), 5)
    M, n = prob.nnodes, 128
    X0 = device(block(M, n, 3), prec, n)
    want = X0.clone()
    for m in (8, n):                                 # kernels loaded, reference block
        few = device(block(M, m, 3), prec, m)
        ctx.cholgs(few)
        ctx.rayleigh_ritz(few)
    ctx.cholgs(want)
    ritz = ctx.rayleigh_ritz(want.clone())
    del few
    ctx.close()
    ctx, _ = context(g, prec, (6, 6, 6), 5)
    X = X0.clone()
    ctx.apply_h(X, torch.empty_like(X))              # tables and coefficients in place

    def starved(room, call):
        torch.cuda.empty_cache()
        hog = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
        try:
            return call()
        finally:
            del hog
            torch.cuda.empty_cache()

    # FP64 blocks take 105 MB, FP32 blocks 53, the digits 185 (Rayleigh-Ritz 369 for its Gram matrix)
    starved(150 << 20, lambda: ctx.cholgs(X))
    err = torch.linalg.vector_norm((X - want).reshape(-1, n), dim=0) / torch.linalg.vector_norm(want.reshape(-1, n), dim=0)
    assert float(err.max()) < (1e-12 if prec == 0 else 2.0 ** -23)
    got = starved(300 << 20, lambda: ctx.rayleigh_ritz(X))
    assert np.abs(got - ritz).max() < (1e-11 if prec == 0 else 1e-6) * np.abs(ritz).max()
    ctx.close()
    # digits that an earlier call left (185 MB) make room for the blocks of a filter (two)
    ctx, _ = context(g, prec, (6, 6, 6), 5)
    ctx.apply_h(X, torch.empty_like(X))
    ctx.cholgs(X0)
    starved(50 << 20, lambda: ctx.filter(X, 2, 2.0, 80.0, -3.0))
    ctx.sync_status()
    ctx.close()


def test_expired_wait_belongs_to_its_context(g):
    """An expired wait of the split products is reported by the synchronous calls of its own context,
    with the block unchanged, until gbc_sync_status has reported it, and by no other context."""
    (a, prob), (b, _) = context(g, 0, (3, 3, 2), 3), context(g, 0, (3, 3, 2), 3)
    X = device(block(prob.nnodes, 20, 3), 0, 20)
    keep = X.clone()
    a.split_wait_selftest()
    b.sync_status()
    Y = X.clone()
    b.cholgs(Y)
    ritz = b.rayleigh_ritz(Y)
    bounds = (2.0, 80.0, -3.0)
    calls = [lambda: a.cholgs(X), lambda: a.rayleigh_ritz(X),
             lambda: a.filter_vjp(X, Y, torch.empty_like(X), 3, *bounds),
             lambda: a.energy_grad(X, np.ones(20), torch.empty_like(X)), a.sync_status]
    for call in calls:
        with pytest.raises(g.GbcError) as e:
            call()
        assert e.value.status == 6                       # GBC_ETIMEOUT
        assert torch.equal(X, keep)
    a.sync_status()                                      # cleared
    a.cholgs(X)
    assert np.abs(a.rayleigh_ritz(X) - ritz).max() < 1e-11 * np.abs(ritz).max()
    a.close()
    b.close()
