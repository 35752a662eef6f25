"""Performance cases of the ChFSI hot path: what a program that solves the
finite-element spinor eigenproblem asks of the library, call by call.

Each case is one public call (or the few calls a program always makes together)
on a seeded problem: mesh, quadrature-point fields, atom-centred projectors and
a spinor block.  Sizes are those of the package's own workloads (6^3 cells at
p = 4 with 32 vectors, 16^3 cells at p = 6 with 256 vectors, slabs with
Dirichlet faces, uneven batches) and odd sizes between them.

``exact`` restates every path in plain torch in 64 bits: dense 1-D operators,
explicit projector tables, gather and scatter by index.
"""
import itertools
import math

import numpy as np
import torch

import paper_2410_02754_gb300 as gbc

# radial channels (width, l): one p channel, or two each of s, p, d
P_CHANNEL = ((0.5, 1),)
SPD_CHANNELS = ((0.5, 0), (0.65, 0), (0.5, 1), (0.65, 1), (0.5, 2), (0.65, 2))
KT = 1.583e-3          # Ha, 500 K

# FP64 operations past which a case has no 64-bit value (about 20 seconds of them)
EXACT_FLOPS = 1.2e13


def _case(name, op, cells, p, nvec, *, dirichlet_z=False, kx=0.0, ky=0.0, kz=0.0, natoms=0,
          spd=True, degree=0, fp32=True, steps=0):
    return dict(name=name, op=op, nx=cells[0], ny=cells[1], nz=cells[2], p=p, nvec=nvec,
                dirichlet_z=dirichlet_z, kx=kx, ky=ky, kz=kz, natoms=natoms, spd=spd,
                degree=degree, fp32=fp32, steps=steps)


def listed():
    return [
        # the smallest call: one H.X on a toy cell in FP64 (unit tests, line searches,
        # a few vectors of a molecule): launch latency
        _case("apply_fp64_tiny", "apply", (3, 2, 2), 3, 5, kx=0.1, ky=-0.2, kz=0.05, natoms=2,
              spd=False, fp32=False),
        # the filter of a small cell: 32 states, many short launches
        _case("filter_small", "filter", (6, 6, 6), 4, 32, natoms=4, spd=False, degree=10),
        # the filter of the flagship workload: 884,736 nodes, 256 spinors, 64 atoms, one k-point
        _case("filter_cube", "filter", (16, 16, 16), 6, 256, kx=0.25, ky=-0.25, natoms=64, degree=20),
        # a slab with Dirichlet faces, odd block width and another order
        _case("filter_slab_odd", "filter", (13, 11, 9), 5, 77, dirichlet_z=True, natoms=14,
              degree=15),
        # the FP64 filter that tight convergence needs
        _case("filter_fp64", "filter", (6, 6, 6), 6, 64, kz=0.25, natoms=6, degree=8, fp32=False),
        # spectrum bounds before the first filter: one vector, FP64
        _case("lanczos_cube", "lanczos", (16, 16, 16), 6, 1, natoms=24, fp32=False, steps=10),
        # orthonormalisation of a filtered FP32 block (mixed-precision cycle)
        _case("cholgs_cube", "cholgs", (16, 16, 16), 6, 256),
        # what follows the filter in every mixed cycle: CholGS, Rayleigh-Ritz, occupations, density
        _case("subspace_mixed", "subspace", (10, 10, 10), 6, 200, kx=0.25, natoms=16),
        # the same in FP64 on a smaller, odd block
        _case("subspace_fp64", "subspace", (9, 8, 7), 4, 75, natoms=5, fp32=False),
        # two-grid start: carry the order-5 block to order 6
        _case("twogrid_cube", "twogrid", (16, 16, 16), 6, 256),
        # gradients through the filter (backward)
        _case("vjp_mid", "vjp", (6, 6, 6), 6, 64, kx=0.25, natoms=8, degree=10),
        # several independent systems of uneven size filtered together
        _case("batch_uneven", "batch", (8, 8, 8), 5, 96, natoms=8, degree=12),
    ]


def draw(rng):
    """A case of the same paths with sizes anywhere in their ranges."""
    op = rng.choice(["apply", "filter", "filter", "filter", "lanczos", "cholgs", "subspace",
                     "subspace", "twogrid", "vjp", "batch"])
    p = rng.choice([3, 4, 5, 6, 6, 7]) if op not in ("vjp", "subspace") else rng.choice([3, 4, 5, 6])
    if op == "twogrid":
        p = rng.choice([3, 4, 5, 6])
    fp32 = op != "lanczos" and rng.random() < (0.5 if op in ("apply", "subspace") else 0.8)
    # cells and vectors log-uniform under a cap on the work of one pass
    cap = {"apply": 2e8, "filter": 1.1e8, "lanczos": 9e5, "cholgs": 1.5e8, "subspace": 4e7,
           "twogrid": 1.5e8, "vjp": 6e6, "batch": 8e6}[op]
    if not fp32 and op != "lanczos":
        cap /= 16
    while True:
        cells = [max(2, round(math.exp(rng.uniform(math.log(3), math.log(16))))) for _ in range(3)]
        nvec = 1 if op == "lanczos" else round(math.exp(rng.uniform(math.log(3), math.log(300))))
        nodes = math.prod(cells) * p ** 3
        if nodes * nvec <= cap and nodes * 2 >= 4 * nvec:
            break
    kpt = op != "batch" and rng.random() < 0.6
    natoms = 0 if op in ("cholgs", "twogrid") else rng.randint(1, max(1, min(40, math.prod(cells) // 40)))
    return dict(op=op, nx=cells[0], ny=cells[1], nz=cells[2], p=p, nvec=nvec,
                dirichlet_z=rng.random() < 0.3, kx=0.25 if kpt else 0.0, ky=0.0,
                kz=rng.choice([0.0, 0.25]) if kpt else 0.0, natoms=natoms, spd=rng.random() < 0.7,
                degree=rng.randint(6, 20) if op in ("filter", "vjp", "batch") else 0, fp32=fp32,
                steps=rng.randint(6, 14) if op == "lanczos" else 0)


# ---------------------------------------------------------------------------------
# problems
# ---------------------------------------------------------------------------------
def _lagrange(nodes, t):
    """Values and derivatives of the Lagrange basis on ``nodes`` at points t: [n, len(t)]."""
    n = len(nodes)
    val, der = np.ones((n, len(t))), np.zeros((n, len(t)))
    for i in range(n):
        others = [m for m in range(n) if m != i]
        for m in others:
            val[i] *= (t - nodes[m]) / (nodes[i] - nodes[m])
            term = np.full(len(t), 1.0 / (nodes[i] - nodes[m]))
            for j in others:
                if j != m:
                    term *= (t - nodes[j]) / (nodes[i] - nodes[j])
            der[i] += term
    return val, der


def _gll(p):
    """Gauss-Lobatto-Legendre nodes and weights of order p on [-1, 1]."""
    leg = np.polynomial.legendre.Legendre.basis(p)
    x = np.concatenate([[-1.0], np.sort(leg.deriv().roots().real), [1.0]])
    for _ in range(3):                       # Newton on (1 - x^2) P_p' inside
        d1, d2 = leg.deriv()(x[1:-1]), leg.deriv(2)(x[1:-1])
        x[1:-1] -= d1 / d2
    x = 0.5 * (x - x[::-1])
    return x, 2.0 / (p * (p + 1) * leg(x) ** 2)


class _Problem:
    """Mesh, fields, projectors of one system, drawn from a seed (1 bohr cells)."""

    def __init__(self, cells, p, periodic, k, natoms, channels, seed, device="cuda"):
        self.ncell, self.p, self.nq = tuple(cells), p, p + 2
        self.periodic = periodic
        self.h = (1.0, 1.0, 1.0)
        self.k = 2.0 * math.pi * np.asarray(k) / np.asarray(cells, np.float64)
        self.nfree = [n * p if per else n * p - 1 for n, per in zip(cells, periodic)]
        self.nnodes = math.prod(self.nfree)
        self.ncells = math.prod(cells)
        rng = np.random.default_rng(1000 + seed)
        box = np.asarray(cells, np.float64)
        # atoms: a jittered lattice away from Dirichlet faces
        per_dim = max(1, math.ceil(natoms ** (1 / 3)))
        sites = np.array(list(itertools.product(range(per_dim), repeat=3)))[:max(natoms, 0)]
        pos = (sites + 0.5 + rng.uniform(-0.1, 0.1, sites.shape)) / per_dim * box
        for d in range(3):
            if not periodic[d]:
                pos[:, d] = box[d] * (0.25 + 0.5 * pos[:, d] / box[d])
        self.pos = pos
        # quadrature points of every cell, [E, nq^3, 3]
        xi, _ = np.polynomial.legendre.leggauss(self.nq)
        t = torch.as_tensor((xi + 1) / 2, device=device)
        ax = [(torch.arange(n, device=device, dtype=torch.float64)[:, None] + t) for n in cells]
        nx, ny, nz = cells
        q = self.nq
        r = torch.empty((nz, ny, nx, q, q, q, 3), dtype=torch.float64, device=device)
        r[..., 0] = ax[0][None, None, :, None, None, :]
        r[..., 1] = ax[1][None, :, None, None, :, None]
        r[..., 2] = ax[2][:, None, None, :, None, None]
        rq = r.reshape(self.ncells, q ** 3, 3)
        boxt = torch.as_tensor(box, device=device)
        pert = torch.as_tensor(periodic, device=device)
        v = torch.zeros(rq.shape[:2], dtype=torch.float64, device=device)
        for R in pos:                                # Gaussian wells, minimum image
            d = rq - torch.as_tensor(R, device=device)
            d = torch.where(pert, d - boxt * torch.round(d / boxt), d)
            v -= 2.0 * torch.exp(-(d * d).sum(-1) / (2 * 0.8 ** 2))
        b = torch.zeros((3,) + tuple(v.shape), dtype=torch.float64, device=device)
        for d in range(3):                           # a few low Fourier modes
            for _ in range(3):
                G = torch.as_tensor(2 * math.pi * rng.integers(-1, 2, 3) / box, device=device)
                b[d] += rng.normal() * torch.cos(rq @ G + rng.uniform(0, 2 * math.pi))
        b *= 0.1 / float((b * b).sum(0).sqrt().max().clamp_min(1e-12))
        self.v, self.b = v, b
        # projectors on the cells (and lattice images) that the ball |r - R - L| < rc meets
        rc = 2.0 if min(cells) >= 4 else 1.2
        self.npj = sum(2 * l + 1 for _, l in channels)
        lo = np.array([[e % nx, (e // nx) % ny, e // (nx * ny)] for e in range(self.ncells)], np.float64)
        images = list(itertools.product(*[(-1, 0, 1) if per else (0,) for per in periodic]))
        self.supp_cell, self.supp_img, self.pvals, self.delta = [], [], [], []
        for R in pos:
            cell, img = [], []
            for L in images:
                c = R + np.asarray(L) * box
                gap = np.maximum(np.maximum(lo - c, 0.0), c - (lo + 1.0))
                hit = np.nonzero((gap * gap).sum(-1) < rc * rc)[0]
                cell.append(hit)
                img.append(np.tile(np.asarray(L, np.int32), (len(hit), 1)))
            cell, img = np.concatenate(cell).astype(np.int32), np.concatenate(img)
            ct = torch.as_tensor(cell, device=device, dtype=torch.long)
            d = rq[ct] - torch.as_tensor(R, device=device) - (
                torch.as_tensor(img, device=device, dtype=torch.float64) * boxt)[:, None, :]
            self.supp_cell.append(cell)
            self.supp_img.append(img)
            self.pvals.append(_projector_values(d, channels, rc))
            A = rng.normal(0, 0.1, (2, 2 * self.npj, 2 * self.npj))
            A = A[0] + 1j * A[1]
            self.delta.append(0.5 * (A + A.conj().T))

    def load(self, ctx):
        ctx.set_mesh(self.ncell, self.h, self.p, self.nq, self.periodic)
        ctx.set_kpoint(self.k)
        ctx.set_fields(self.v.cpu().numpy(), *[x.cpu().numpy() for x in self.b])
        n = len(self.pos)
        if n:
            ctx.set_projectors(n, [self.npj] * n, [len(c) for c in self.supp_cell],
                               np.concatenate(self.supp_cell), np.concatenate(self.supp_img),
                               torch.cat([x.reshape(-1) for x in self.pvals]).cpu().numpy(),
                               np.concatenate([d.reshape(-1) for d in self.delta]))

    def bounds(self):
        """(lT, lmax, lmin) around the spectrum of M_D^-1 H: the 1-D kinetic maximum per
        direction plus the potential and projector ranges; lT where a block of low states ends."""
        x, w = _gll(self.p)
        xq, wq = np.polynomial.legendre.leggauss(self.nq)
        _, D = _lagrange(x, xq)
        s = 1.0 / np.sqrt(w)
        top = np.linalg.eigvalsh(s[:, None] * ((D * wq) @ D.T) * s)[-1] * 2.0     # (2/h)^2 / 2, h = 1
        lmax = 3.0 * top * 1.05 + 12.0
        return 0.06 * lmax, lmax, -6.0


def _projector_values(d, channels, rc):
    """r^l exp(-r^2 / 2 s^2) Y_lm, normalised on [0, rc], at the offsets d [..., 3]."""
    r = d.norm(dim=-1)
    u = d / r.clamp_min(1e-14)[..., None]
    x, y, z = u.unbind(-1)
    t = np.linspace(0.0, rc, 4001)
    cols = []
    for s, l in channels:
        f = (t ** l * np.exp(-t * t / (2 * s * s))) ** 2 * t * t
        norm = 1.0 / math.sqrt(float(((f[1:] + f[:-1]) / 2).sum() * (t[1] - t[0])))
        rad = norm * r ** l * torch.exp(-r * r / (2 * s * s)) * (r < rc)
        if l == 0:
            cols.append(rad * 0.5 / math.sqrt(math.pi))
        elif l == 1:
            cols += [math.sqrt(3 / (4 * math.pi)) * rad * c for c in (y, z, x)]
        else:
            a, b, c = 0.5 * math.sqrt(15 / math.pi), 0.25 * math.sqrt(5 / math.pi), 0.25 * math.sqrt(15 / math.pi)
            cols += [a * rad * x * y, a * rad * y * z, b * rad * (3 * z * z - 1), a * rad * x * z,
                     c * rad * (x * x - y * y)]
    return torch.stack(cols, dim=-1)


def _problem(case, seed, p=None, cells=None):
    cells = cells or (case["nx"], case["ny"], case["nz"])
    return _Problem(cells, p or case["p"], (True, True, not case["dirichlet_z"]),
                    (case["kx"], case["ky"], case["kz"]), case["natoms"],
                    SPD_CHANNELS if case["spd"] else P_CHANNEL, seed)


def _systems(case, seed):
    """The systems of a batch: (problem, nvec, degree), uneven around the case's sizes."""
    out = []
    for i, (dn, dp, fv, dd) in enumerate(((0, 0, 1.0, 0), (1, -1, 0.75, 3), (-1, 1, 0.55, -2), (0, 0, 1.3, 1))):
        cells = tuple(max(2, case[d] + dn) for d in ("nx", "ny", "nz"))
        p = min(7, max(2, case["p"] + dp))
        out.append((_problem(case, seed * 10 + i, p, cells), max(1, int(case["nvec"] * fv)),
                    max(2, case["degree"] + dd)))
    return out


def _block(nnodes, nvec, seed, fp32):
    """Random spinor block [M, 2, nvec], real and imaginary parts uniform in [-1, 1)."""
    g = torch.Generator(device="cuda").manual_seed(7919 * seed + 17)
    x = torch.rand((nnodes, 2, nvec, 2), generator=g, device="cuda", dtype=torch.float32)
    x = torch.view_as_complex(x.mul_(2).sub_(1))
    return x if fp32 else x.to(torch.complex128)


def _subspace_block(prob, nvec, seed, fp32):
    """A block as a filter leaves it: columns that overlap and differ in size, amplitudes
    that fall off away from the middle of the cell."""
    x = _block(prob.nnodes, nvec, seed, True)
    z = torch.linspace(-1, 1, prob.nfree[2], device="cuda")
    env = torch.exp(-6.0 * z * z).repeat_interleave(prob.nfree[0] * prob.nfree[1])
    x *= env[:, None, None]
    x[:, :, 1:] += 0.4 * x[:, :, :-1].clone()
    x *= torch.logspace(0, -2, nvec, device="cuda")
    return x if fp32 else x.to(torch.complex128)


# ---------------------------------------------------------------------------------
# the measured calls
# ---------------------------------------------------------------------------------
def _context(prob, fp32):
    ctx = gbc.Context(torch.cuda.current_device())
    prob.load(ctx)
    ctx.set_precision(gbc.FP32 if fp32 else gbc.FP64)
    return ctx


def prepare(case, seed):
    op, fp32, nvec = case["op"], case["fp32"], case["nvec"]
    if op == "batch":
        sysm = _systems(case, seed)
        ctxs = [_context(prob, fp32) for prob, _, _ in sysm]
        blocks = [_block(prob.nnodes, n, 31 * seed + i, fp32) for i, (prob, n, _) in enumerate(sysm)]
        if fp32:
            for c, x in zip(ctxs, blocks):
                c.tune(x.shape[2])
        return dict(op=op, ctxs=ctxs, X0=blocks, X=[torch.empty_like(x) for x in blocks],
                    degrees=[d for _, _, d in sysm], bounds=[prob.bounds() for prob, _, _ in sysm],
                    batch=gbc.Batch(ctxs), stream=torch.cuda.Stream())
    prob = _problem(case, seed)
    ctx = _context(prob, fp32)
    st = dict(op=op, ctx=ctx, degree=case["degree"], bounds=prob.bounds(), steps=case["steps"])
    if op == "apply":
        st["X"] = _block(prob.nnodes, nvec, seed, fp32)
        st["Y"] = torch.empty_like(st["X"])
    elif op == "filter":
        if fp32:
            ctx.tune(nvec)
        st["X0"] = _block(prob.nnodes, nvec, seed, fp32)
        st["X"] = torch.empty_like(st["X0"])
    elif op == "lanczos":
        st["v0"] = _block(prob.nnodes, 1, seed, False).reshape(prob.nnodes, 2)
    elif op in ("cholgs", "subspace"):
        st["X0"] = _subspace_block(prob, nvec, seed, fp32)
        st["X"] = torch.empty_like(st["X0"])
        st["nelec"] = max(1, nvec // 2)
        st["dens"] = torch.empty((prob.ncells, 4, prob.nq ** 3), dtype=torch.float64, device="cuda")
    elif op == "twogrid":
        coarse = _problem(dict(case, natoms=0), seed, case["p"] - 1)
        st["coarse"] = _context(coarse, fp32)
        st["X"] = _block(coarse.nnodes, nvec, seed, fp32)
        st["Y"] = torch.empty((prob.nnodes, 2, nvec), dtype=st["X"].dtype, device="cuda")
    elif op == "vjp":
        if fp32:
            ctx.tune(nvec)
        st["X"] = _block(prob.nnodes, nvec, seed, fp32)
        st["GY"] = _block(prob.nnodes, nvec, seed + 5000, fp32)
        st["GX"] = torch.empty_like(st["X"])
    return st


def run(st):
    op = st["op"]
    if op == "batch":
        for x, x0 in zip(st["X"], st["X0"]):
            x.copy_(x0)
        st["stream"].wait_stream(torch.cuda.current_stream())
        st["batch"].filter(st["X"], st["degrees"], st["bounds"], st["stream"])
        torch.cuda.current_stream().wait_stream(st["stream"])
        return st["X"]
    ctx = st["ctx"]
    if op == "apply":
        ctx.apply_h(st["X"], st["Y"])
        return st["Y"]
    if op == "filter":
        st["X"].copy_(st["X0"])
        ctx.filter(st["X"], st["degree"], *st["bounds"])
        return st["X"]
    if op == "lanczos":
        return ctx.lanczos_bounds(st["v0"], st["steps"])
    if op == "cholgs":
        st["X"].copy_(st["X0"])
        ctx.cholgs(st["X"])
        return st["X"]
    if op == "subspace":
        # Ritz vectors are unique up to phases; the density made from them is unique
        st["X"].copy_(st["X0"])
        ctx.cholgs(st["X"])
        ritz = ctx.rayleigh_ritz(st["X"])
        occ, _ = gbc.fermi_occupations(ritz[None], None, st["nelec"], KT)
        ctx.density_dev(st["X"], torch.from_numpy(occ[0]).cuda(), st["dens"])
        return {"ritz": ritz, "density": st["dens"]}
    if op == "twogrid":
        ctx.prolongate_from(st["coarse"], st["X"], st["Y"])
        return st["Y"]
    gV, gBx, gBy, gBz, gD = ctx.filter_vjp(st["X"], st["GY"], st["GX"], st["degree"], *st["bounds"])
    return {"gX": st["GX"], "gV": gV, "gB": [gBx, gBy, gBz], "gDelta": gD}


# ---------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------
def _sizes(case, p=None, cells=None):
    cells = cells or (case["nx"], case["ny"], case["nz"])
    p = p or case["p"]
    M = cells[0] * p * cells[1] * p * (cells[2] * p - (1 if case["dirichlet_z"] else 0))
    return math.prod(cells), M, p + 1, p + 2


def _hx_flops(E, n, q, nvec, kpt, natoms, spd):
    """One H.X: even-odd sum factorisation on complex data, two spins, plus projectors."""
    eo = lambda no, ni: 2 * (no * ni + no + ni)          # real flop of an even-odd product, x 2 parts
    g = eo(n, n) * (2 if kpt else 1)
    kin = n * n * (4 * eo(n, n) + 3 * g)
    pot = 2 * (n * n * eo(q, n) + n * q * eo(q, n) + q * q * eo(q, n))
    npj = 18 if spd else 3
    support = natoms * 60 * (n - 1) ** 3
    return nvec * (E * (2 * (kin + pot) + 28 * q ** 3) + 2 * 2 * 8 * support * npj)


def _filter_work(case, p=None, cells=None, nvec=None, degree=None):
    E, M, n, q = _sizes(case, p, cells)
    nvec, degree = nvec or case["nvec"], degree or case["degree"]
    kpt = bool(case["kx"] or case["ky"] or case["kz"])
    el = 8 if case["fp32"] else 16
    return (2 * M * 2 * nvec * el + E * 4 * q ** 3 * el / 2,
            degree * (_hx_flops(E, n, q, nvec, kpt, case["natoms"], case["spd"]) + 20 * M * nvec))


def work(case):
    op, nvec = case["op"], case["nvec"]
    E, M, n, q = _sizes(case)
    el = 8 if case["fp32"] else 16
    block = M * 2 * nvec * el
    kpt = bool(case["kx"] or case["ky"] or case["kz"])
    hx = _hx_flops(E, n, q, nvec, kpt, case["natoms"], case["spd"])
    fields = E * 4 * q ** 3 * el / 2
    if op == "apply":
        b, f = 2 * block + fields, hx
    elif op == "filter":
        b, f = _filter_work(case)
    elif op == "batch":
        b = f = 0
        for dn, dp, fv, dd in ((0, 0, 1.0, 0), (1, -1, 0.75, 3), (-1, 1, 0.55, -2), (0, 0, 1.3, 1)):
            cells = tuple(max(2, case[d] + dn) for d in ("nx", "ny", "nz"))
            w = _filter_work(case, min(7, max(2, case["p"] + dp)), cells,
                             max(1, int(nvec * fv)), max(2, case["degree"] + dd))
            b, f = b + w[0], f + w[1]
    elif op == "lanczos":
        b, f = block + fields, case["steps"] * (hx + 16 * 2 * M * case["steps"])
    elif op == "cholgs":
        b, f = 2 * block, 12 * 2 * M * nvec * nvec
    elif op == "subspace":
        b, f = 2 * block + E * 4 * q ** 3 * 8, 24 * 2 * M * nvec * nvec + 2 * hx
    elif op == "twogrid":
        _, Mc, _, _ = _sizes(case, case["p"] - 1)
        c = n - 1
        b, f = (M + Mc) * 2 * nvec * el, E * nvec * 2 * 4 * c * n * (c * c + c * n + n * n)
    else:
        b, f = 3 * block + 2 * fields, 3 * case["degree"] * hx
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------------
# 64-bit values in plain torch
# ---------------------------------------------------------------------------------
class _Reference:
    """The FE Hamiltonian of one _Problem, complex128, dense 1-D operators."""

    def __init__(self, prob):
        self.pr, p, q = prob, prob.p, prob.nq
        dev = "cuda"
        x, w = _gll(p)
        xq, wq = np.polynomial.legendre.leggauss(q)
        N, D = _lagrange(x, xq)
        B, A, C = (N * wq) @ N.T, (D * wq) @ D.T, (N * wq) @ D.T
        to = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=dev, dtype=torch.complex128)
        self.N = to(N)
        self.B = to(B / 2)                                                  # h = 1
        self.G = [to(A - 0.5j * k * (C - C.T)) for k in prob.k]
        idx, md = [], []
        for n, per in zip(prob.ncell, prob.periodic):
            g = np.arange(n)[:, None] * p + np.arange(p + 1)
            m = np.zeros(n * p + 1)
            np.add.at(m, g, np.broadcast_to(w / 2, g.shape))
            if per:
                m[0] += m[-1]
                md.append(m[:-1])
                idx.append(g % (n * p))
            else:
                md.append(m[1:-1])
                idx.append(np.where((g == 0) | (g == n * p), -1, g - 1))
        gx, gy, gz = [torch.as_tensor(a, device=dev) for a in idx]
        nfx, nfy = prob.nfree[0], prob.nfree[1]
        I = ((gz[:, None, None, :, None, None] * nfy + gy[None, :, None, None, :, None]) * nfx
             + gx[None, None, :, None, None, :])
        ok = ((gz >= 0)[:, None, None, :, None, None] & (gy >= 0)[None, :, None, None, :, None]
              & (gx >= 0)[None, None, :, None, None, :])
        self.idx = torch.where(ok, I, prob.nnodes).reshape(prob.ncells, -1)   # nnodes = the zero row
        mx, my, mz = [torch.as_tensor(m, device=dev) for m in md]
        self.md = (mz[:, None, None] * my[:, None] * mx).reshape(-1)
        t = torch.as_tensor((xq + 1) / 2, device=dev)
        self.wj = torch.as_tensor((wq[:, None, None] * wq[:, None] * wq).reshape(-1) / 8, device=dev)
        self.V, self.Bf = prob.v, prob.b
        # projector tables on each atom's distinct nodes
        self.atoms = []
        c = torch.arange(prob.ncells, device=dev)
        nx, ny = prob.ncell[0], prob.ncell[1]
        org = torch.stack([c % nx, (c // nx) % ny, c // (nx * ny)], -1).double()
        pts = torch.stack(torch.meshgrid(t, t, t, indexing="ij")[::-1], -1).reshape(-1, 3)
        kk, box = torch.as_tensor(prob.k, device=dev), torch.as_tensor(np.asarray(prob.ncell, float), device=dev)
        for cell, img, pv, dl in zip(prob.supp_cell, prob.supp_img, prob.pvals, prob.delta):
            ce = torch.as_tensor(cell, device=dev, dtype=torch.long)
            r = org[ce][:, None, :] + pts - (torch.as_tensor(img, device=dev).double() * box)[:, None, :]
            f = (self.wj * torch.exp(-1j * (r @ kk)))[..., None] * pv
            f = f.reshape(len(cell), q, q, q, -1)
            for axis in ("iq,eqrsc->eirsc", "iq,erqsc->erisc", "iq,ersqc->ersic"):
                f = torch.einsum(axis, self.N, f)
            nodes, inv = torch.unique(self.idx[ce], return_inverse=True)
            P = torch.zeros((len(nodes), pv.shape[-1]), dtype=torch.complex128, device=dev)
            P.index_add_(0, inv.reshape(-1), f.reshape(-1, pv.shape[-1]))
            P[nodes == prob.nnodes] = 0
            self.atoms.append((nodes, P, torch.as_tensor(dl, device=dev)))

    def cells(self, X):
        """[E, nz, ny, nx, 2 * nvec] nodal values of every cell."""
        n = self.pr.p + 1
        X = torch.cat([X.reshape(self.pr.nnodes, -1), X.new_zeros((1, X[0].numel()))])
        return X[self.idx].reshape(self.pr.ncells, n, n, n, -1)

    def gauss(self, Xc):
        N = self.N
        Xc = torch.einsum("kq,ejikm->ejiqm", N, Xc)
        Xc = torch.einsum("kq,ejkim->ejqim", N, Xc)
        return torch.einsum("kq,ekjim->eqjim", N, Xc)

    def apply(self, X, V=None, Bf=None, deltas=None):
        pr = self.pr
        nvec, q, n = X.shape[2], pr.nq, pr.p + 1
        V, Bf = self.V if V is None else V, self.Bf if Bf is None else Bf
        Xc = self.cells(X)
        B, (Gx, Gy, Gz), N = self.B, self.G, self.N
        ap = {0: "ik,ejlkm->ejlim", 1: "ik,ejklm->ejilm", 2: "ik,ekjlm->eijlm"}
        bx, by = torch.einsum(ap[0], B, Xc), torch.einsum(ap[1], B, Xc)
        out = torch.einsum(ap[2], B, torch.einsum(ap[1], B, torch.einsum(ap[0], Gx, Xc)))
        out = out + torch.einsum(ap[2], B, torch.einsum(ap[1], Gy, bx))
        out = out + torch.einsum(ap[2], Gz, torch.einsum(ap[0], B, by))
        U = self.gauss(Xc).reshape(pr.ncells, q ** 3, 2, nvec)
        k2 = 0.5 * float((pr.k ** 2).sum())
        w = self.wj
        d, bx_, by_, bz_ = [(w * f)[..., None] for f in (V + k2, Bf[0], Bf[1], Bf[2])]
        up, dn = U[:, :, 0], U[:, :, 1]
        W = torch.stack([(d + bz_) * up + (bx_ - 1j * by_) * dn,
                         (bx_ + 1j * by_) * up + (d - bz_) * dn], 2)
        W = W.reshape(pr.ncells, q, q, q, 2 * nvec)
        for k in (0, 1, 2):
            W = torch.einsum(ap[k], N, W)
        out = out + W
        Y = torch.zeros((pr.nnodes + 1, 2 * nvec), dtype=X.dtype, device=X.device)
        Y = Y.index_add(0, self.idx.reshape(-1), out.reshape(-1, 2 * nvec))[:-1]
        Y = Y.reshape(pr.nnodes, 2, nvec)
        for a, (nodes, P, dl) in enumerate(self.atoms):
            keep = nodes < pr.nnodes
            nd, Pk = nodes[keep], P[keep]
            D = dl if deltas is None else deltas[a]
            C = torch.einsum("jc,jsv->csv", Pk.conj(), X[nd]).reshape(-1, nvec)
            C = (D @ C).reshape(-1, 2, nvec)
            Y = Y.index_add(0, nd, torch.einsum("jc,csv->jsv", Pk, C))
        return Y

    def filter(self, X, m, lT, lmax, lmin, **kw):
        c, e = 0.5 * (lmax + lT), 0.5 * (lmax - lT)
        s1 = e / (lmin - c)
        inv = (1.0 / self.md)[:, None, None]
        sig, prev = s1, X
        cur = (inv * self.apply(X, **kw) - c * X) * (s1 / e)
        for _ in range(1, m):
            s2 = 1.0 / (2.0 / s1 - sig)
            cur, prev = (inv * self.apply(cur, **kw) - c * cur) * (2 * s2 / e) - sig * s2 * prev, cur
            sig = s2
        return cur

    def chunk(self, copies=14):
        """Vectors at a time so that the temporaries of an apply fit 40 GB."""
        return max(1, int(40e9 / (copies * self.pr.ncells * (self.pr.nq ** 3) * 2 * 16)))


def _mesh_only(prob):
    """The problem without its atoms (mesh only)."""
    out = object.__new__(_Problem)
    out.__dict__.update(prob.__dict__, supp_cell=[], supp_img=[], pvals=[], delta=[])
    return out


def _over_columns(ref, X, fn, copies=14):
    step = ref.chunk(copies)
    return torch.cat([fn(X[:, :, i:i + step]) for i in range(0, X.shape[2], step)], 2)


def _occupations(e, nelec):
    lo, hi = e.min() - 1.0, e.max() + 1.0
    f = lambda mu: 1.0 / (1.0 + np.exp(np.clip((e - mu) / KT, -700, 700)))
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if f(mid).sum() < nelec else (lo, mid)
    return f(0.5 * (lo + hi))


def _exact_filter(prob, X, degree):
    ref = _Reference(prob)
    return _over_columns(ref, X.to(torch.complex128), lambda x: ref.filter(x, degree, *prob.bounds()))


@torch.no_grad()
def _exact_plain(case, seed):
    op, nvec, fp32 = case["op"], case["nvec"], case["fp32"]
    if op == "batch":
        return [_exact_filter(prob, _block(prob.nnodes, n, 31 * seed + i, fp32), d)
                for i, (prob, n, d) in enumerate(_systems(case, seed))]
    prob = _problem(case, seed)
    if op == "filter":
        return _exact_filter(prob, _block(prob.nnodes, nvec, seed, fp32), case["degree"])
    if op == "twogrid":
        coarse = _problem(dict(case, natoms=0), seed, case["p"] - 1)
        X = _block(coarse.nnodes, nvec, seed, fp32).to(torch.complex128)
        T = torch.as_tensor(_lagrange(_gll(coarse.p)[0], _gll(prob.p)[0])[0], device="cuda",
                            dtype=torch.complex128)
        rc, rf = _Reference(coarse), _Reference(_mesh_only(prob))

        def carry(x):
            c = rc.cells(x)
            c = torch.einsum("iq,ejlim->ejlqm", T, c)
            c = torch.einsum("iq,ejilm->ejqlm", T, c)
            c = torch.einsum("iq,eijlm->eqjlm", T, c)
            out = torch.zeros((prob.nnodes + 1, c.shape[-1]), dtype=x.dtype, device="cuda")
            out[rf.idx.reshape(-1)] = c.reshape(-1, c.shape[-1])
            return out[:-1].reshape(prob.nnodes, 2, -1)
        return _over_columns(rf, X, carry, 4)
    ref = _Reference(prob)
    if op == "apply":
        X = _block(prob.nnodes, nvec, seed, fp32).to(torch.complex128)
        return _over_columns(ref, X, ref.apply)
    if op == "lanczos":
        v = _block(prob.nnodes, 1, seed, False)
        md = ref.md[:, None, None]
        dot = lambda a, b: complex((md * a.conj() * b).sum())
        V, al, be = [v / math.sqrt(dot(v, v).real)], [], []
        for _ in range(case["steps"]):
            w = ref.apply(V[-1]) / md
            al.append(dot(V[-1], w).real)
            for _ in range(2):
                for u in V:
                    w = w - dot(u, w) * u
            be.append(math.sqrt(max(dot(w, w).real, 0.0)))
            V.append(w / be[-1])
        ev = np.linalg.eigvalsh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))
        return float(ev[0]), float(ev[-1] + be[-1])
    X = _subspace_block(prob, nvec, seed, fp32).to(torch.complex128)
    flat = X.reshape(-1, nvec)
    m2 = ref.md.repeat_interleave(2)[:, None]
    L = torch.linalg.cholesky(flat.mH @ (m2 * flat))
    flat = torch.linalg.solve_triangular(L.mH, flat, upper=True, left=False)
    X = flat.reshape(prob.nnodes, 2, nvec)
    if op == "cholgs":
        return X
    HX = _over_columns(ref, X, ref.apply).reshape(-1, nvec)
    Hp = flat.mH @ HX
    ev, Q = torch.linalg.eigh(0.5 * (Hp + Hp.mH))
    X = (flat @ Q).reshape(prob.nnodes, 2, nvec)
    occ = torch.as_tensor(_occupations(ev.cpu().numpy(), max(1, nvec // 2)), device="cuda")
    dens = 0
    step = ref.chunk(6)
    for i in range(0, nvec, step):
        U = ref.gauss(ref.cells(X[:, :, i:i + step])).reshape(prob.ncells, prob.nq ** 3, 2, -1)
        u, d, f = U[:, :, 0], U[:, :, 1], occ[i:i + step]
        uu, dd, ud = (u.abs() ** 2 * f).sum(-1), (d.abs() ** 2 * f).sum(-1), (u.conj() * d * f).sum(-1)
        dens = dens + torch.stack([uu + dd, 2 * ud.real, 2 * ud.imag, uu - dd], 1)
    return {"ritz": ev.cpu().numpy(), "density": dens}


def _exact_vjp(case, seed):
    prob = _problem(case, seed)
    ref = _Reference(prob)
    nvec, fp32 = case["nvec"], case["fp32"]
    X = _block(prob.nnodes, nvec, seed, fp32).to(torch.complex128)
    GY = _block(prob.nnodes, nvec, seed + 5000, fp32).to(torch.complex128)
    V = ref.V.clone().requires_grad_()
    B = ref.Bf.clone().requires_grad_()
    D = [dl.clone().requires_grad_() for _, _, dl in ref.atoms]
    gX = []
    step = max(1, ref.chunk(30 * case["degree"]))
    for i in range(0, nvec, step):
        x = X[:, :, i:i + step].clone().requires_grad_()
        y = ref.filter(x, case["degree"], *prob.bounds(), V=V, Bf=B, deltas=D)
        y.backward(GY[:, :, i:i + step].contiguous())
        gX.append(x.grad)
    gD = torch.cat([(0.5 * (d.grad + d.grad.mH)).reshape(-1) for d in D]) if D else torch.zeros(0)
    return {"gX": torch.cat(gX, 2), "gV": V.grad, "gB": list(B.grad), "gDelta": gD}


def exact(case, seed):
    """What run() returns, in 64 bits, or None where that takes too long."""
    # dense complex products against even-odd real ones: about 3 times the operations
    cost = work(case)["flops"] * {"subspace": 1, "cholgs": 1, "vjp": 9}.get(case["op"], 3)
    if cost > EXACT_FLOPS:
        return None
    out = _exact_vjp(case, seed) if case["op"] == "vjp" else _exact_plain(case, seed)
    torch.cuda.empty_cache()
    return out
