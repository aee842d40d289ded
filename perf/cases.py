"""Performance cases of the hp-DG solver: what its users have it do, through the C ABI's Python binding.

Four kinds of pass, each one call of a public entry point on handles that a program makes once per mesh:

  solve    dg_pcg_solve       preconditioned CG for one load vector, the framework's main call
  apply    dg_apply           y = A x, the matrix-free operator alone (time stepping, other Krylov methods)
  precond  dg_precond_apply   z = B r, the subspace-correction preconditioner alone, in FP64
  batch    Batch.solve        many uneven problems x several load vectors in one launch

The mesh belongs to the case, the vectors to the seed. Loads are sums of four random sine modes (the repository's
workloads); solves run to a relative residual of 1e-10, the tolerance of its conforming workload.

`exact` assembles the same forms by plain Gauss quadrature in torch, in 64 bits, sharing no code with the package.
"""
import functools
import math

import numpy as np
import torch

from paper_2009_01287_gb300 import binding as B
from paper_2009_01287_gb300 import inputs

RTOL, MAXIT = 1e-10, 2000
QUAD = inputs.QUADRILATERAL


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one small conforming Poisson problem, exact coarse solve: the 8x8 p = 2 workload, all latency
        dict(name="solve 2D conforming p2", kind="solve", dim=2, base=8, depth=0, prob=0.0, pmin=2, pmax=2, mesh=0,
             domain="box", form="sipg", eta=22.5, prec="fp64", lor="exact", contrast=1.0),
        # a step of an adaptive sequence: a few thousand unknowns on the L-shaped domain
        dict(name="solve 2D L-shape", kind="solve", dim=2, base=6, depth=3, prob=0.35, pmin=1, pmax=6, mesh=1,
             domain="lshape", form="sipg", eta=0.0, prec="mixed", lor="amg", contrast=1.0),
        # the 2D hp-random benchmark workload, 98k unknowns, mixed precision
        dict(name="solve 2D hp", kind="solve", dim=2, base=32, depth=3, prob=0.3, pmin=1, pmax=6, mesh=0,
             domain="box", form="sipg", eta=0.0, prec="mixed", lor="amg", contrast=1.0),
        # the same recipe with BR2, a jumping coefficient and plain FP64
        dict(name="solve 2D hp BR2 coef FP64", kind="solve", dim=2, base=23, depth=3, prob=0.3, pmin=1, pmax=6, mesh=3,
             domain="box", form="br2", eta=0.0, prec="fp64", lor="amg", contrast=20.0),
        # curved elements
        dict(name="solve 2D curved", kind="solve", dim=2, base=16, depth=3, prob=0.3, pmin=1, pmax=6, mesh=4,
             domain="curved", form="sipg", eta=0.0, prec="mixed", lor="amg", contrast=1.0),
        # the 3D hp-random recipe (BR2, mixed) on a 10^3 base, 430k unknowns
        dict(name="solve 3D hp BR2", kind="solve", dim=3, base=10, depth=2, prob=0.2, pmin=1, pmax=5, mesh=0,
             domain="box", form="br2", eta=0.0, prec="mixed", lor="amg", contrast=1.0),
        # many uneven problems with several loads each
        dict(name="batch 2D hp", kind="batch", problems=24, rhs=3, base_lo=4, base_hi=20, depth=3, prob=0.3,
             pmin=1, pmax=8, mesh=7),
        # the operator on a large 2D mesh of all degrees
        dict(name="apply 2D hp large", kind="apply", dim=2, base=64, depth=3, prob=0.3, pmin=1, pmax=8, mesh=5,
             domain="box", form="sipg", eta=0.0, contrast=1.0),
        # the operator on mapped quadrilaterals, the benchmark mesh
        dict(name="apply 2D mapped", kind="apply", dim=2, base=32, depth=3, prob=0.3, pmin=1, pmax=6, mesh=0,
             domain="quad", form="sipg", eta=0.0, contrast=1.0),
        # the operator on a middle-sized cube mesh, SIPG, jumping coefficient, odd base
        dict(name="apply 3D hp SIPG coef", kind="apply", dim=3, base=5, depth=2, prob=0.2, pmin=1, pmax=6, mesh=2,
             domain="box", form="sipg", eta=0.0, contrast=20.0),
        # the operator of the 3D hp-random benchmark workload, 1.7M unknowns
        dict(name="apply 3D hp BR2 large", kind="apply", dim=3, base=16, depth=2, prob=0.2, pmin=1, pmax=5, mesh=0,
             domain="box", form="br2", eta=0.0, contrast=1.0),
        # the preconditioner alone on a cube mesh, FP64
        dict(name="precond 3D hp FP64", kind="precond", dim=3, base=7, depth=2, prob=0.2, pmin=1, pmax=5, mesh=6,
             domain="box", form="br2", eta=0.0, prec="fp64", lor="amg", contrast=1.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    mesh = rng.randrange(1000)
    kind = rng.choice(["solve", "solve", "solve", "apply", "apply", "precond", "batch"])
    if kind == "batch":
        return dict(kind=kind, problems=_log_int(rng, 2, 24), rhs=rng.randint(1, 3), base_lo=4,
                    base_hi=rng.randint(6, 20), depth=rng.randint(1, 3), prob=0.3, pmin=1, pmax=rng.randint(2, 8),
                    mesh=mesh)
    dim = rng.choice([2, 2, 3])
    c = dict(kind=kind, dim=dim, depth=rng.randint(1, 4 - dim + 1), prob=0.3 if dim == 2 else 0.2, mesh=mesh,
             domain="box", form=rng.choice(["sipg", "br2"]), eta=0.0, contrast=rng.choice([1.0, 1.0, 20.0]))
    c["pmin"] = rng.randint(1, 3)
    if dim == 2:
        top = 64 if kind == "apply" else 32
        c["base"] = _log_int(rng, 3, top)
        c["pmax"] = rng.randint(max(c["pmin"], 2), 8 if c["base"] <= top // 2 else 6)
        c["domain"] = rng.choice(["box", "box", "quad", "curved", "lshape"]) if c["base"] <= 32 else "box"
        if c["domain"] == "lshape":
            c["base"] += c["base"] % 2
    else:
        c["base"] = _log_int(rng, 2, {"apply": 12, "solve": 7, "precond": 6}[kind])
        c["pmax"] = rng.randint(max(c["pmin"], 2), 6 if c["base"] <= 5 else 5)
        if c["base"] > 5:
            c["pmin"] = 1
    if kind != "apply":
        c["prec"] = "fp64" if kind == "precond" else rng.choice(["mixed", "mixed", "fp64"])
        c["lor"] = "exact" if _dofs([_mesh(c)])[0] <= 3000 and rng.random() < 0.5 else "amg"
    return c


# ------------------------------------------------------------------ meshes
def _mesh(c):
    if c["depth"] == 0 and c["pmin"] == c["pmax"]:
        m = inputs.uniform_mesh(c["dim"], c["base"], c["pmin"])
    else:
        m = inputs.random_refined_mesh(c["dim"], c["base"], c["depth"], c["prob"], c["pmin"], c["pmax"], c["mesh"])
    if c["domain"] == "lshape":
        m = inputs.lshape(m)
    elif c["domain"] == "quad":
        m = inputs.with_corners(m, QUAD)
    elif c["domain"] == "curved":
        m = inputs.with_mapping(m, inputs.WavyMap())
    if c.get("contrast", 1.0) != 1.0:
        m = inputs.with_coeff(m, inputs.base_parity_coeff(m, c["base"], (1.0, c["contrast"])))
    return m


def _batch_meshes(c):
    rng = np.random.Generator(np.random.PCG64(c["mesh"]))
    span = math.log(c["base_lo"]), math.log(c["base_hi"])
    return [inputs.random_refined_mesh(2, int(round(math.exp(rng.uniform(*span)))), c["depth"], c["prob"], c["pmin"],
                                       c["pmax"], 1000 * c["mesh"] + k) for k in range(c["problems"])]


def _options(c):
    return B.make_options(form=B.DG_FORM_BR2 if c.get("form") == "br2" else B.DG_FORM_SIPG, eta=c.get("eta", 0.0),
                          precision=B.DG_PREC_FP64 if c.get("prec") == "fp64" else B.DG_PREC_MIXED,
                          lor=B.DG_LOR_EXACT if c.get("lor") == "exact" else B.DG_LOR_AMG)


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _vector(n, seed):
    return torch.from_numpy(np.random.Generator(np.random.PCG64(seed)).standard_normal(n)).to(_device())


def _dofs(meshes):
    return [int(((m.p.astype(np.int64) + 1) ** m.dim).sum()) for m in meshes]


def _loads(c, seed):
    """The load vectors of a solve (one) or of a batch (rhs per problem), one after another."""
    if c["kind"] == "batch":
        meshes = _batch_meshes(c)
        return torch.cat([_load(m, seed * 100003 + k * c["rhs"] + r)
                          for k, m in enumerate(meshes) for r in range(c["rhs"])])
    return _load(_mesh(c), seed)


# ------------------------------------------------------------------ a pass
def prepare(case, seed):
    if case["kind"] == "batch":
        batch = B.Batch(_batch_meshes(case), n_rhs=case["rhs"])
        b = _loads(case, seed)
        return dict(kind="batch", batch=batch, b=b, x=torch.empty_like(b))
    mesh = B.Mesh(_mesh(case), _options(case))
    pc = B.Precond(mesh) if case["kind"] != "apply" else None
    b = _loads(case, seed) if case["kind"] == "solve" else _vector(mesh.n_dofs, seed)
    return dict(kind=case["kind"], mesh=mesh, pc=pc, b=b, x=torch.empty_like(b))


def run(state):
    b, x = state["b"], state["x"]
    s = torch.cuda.current_stream()
    if state["kind"] == "solve":
        B.dg_pcg_solve(state["mesh"].h, state["pc"].h, b, x, RTOL, MAXIT, s)
    elif state["kind"] == "batch":
        state["batch"].solve(b, x, RTOL, MAXIT, s)
    elif state["kind"] == "apply":
        B.dg_apply(state["mesh"].h, b, x, s)
    else:
        B.dg_precond_apply(state["pc"].h, b, x, s)
    return x


# ------------------------------------------------------------------ what a pass cannot do without
def _apply_work(m):
    """One y = A x: x read and y written, per element its degree, offset and scales (24 B) and per touching pair its
    indices and penalty (16 B). Operations: the volume term sum-factorised (two 1D products per direction in 2D, the
    mass and stiffness products of the three directions shared in 3D), and per pair of touching elements the value
    and flux traces of both sides carried to the other and back, with the 1D tables of the smaller degree."""
    n = m.p.astype(np.float64) + 1
    d = m.dim
    flops = float((2 * (2 * d if d == 2 else 7) * n ** (d + 1)).sum())
    pairs = 0
    for _, left, right, _, _ in _touching(m):
        q = np.where(right >= 0, np.minimum(n[left], n[np.maximum(right, 0)]), n[left])
        flops += float((2 * 8 * (d - 1) * q ** d).sum())
        pairs += len(left)
    dofs = float((n ** d).sum())
    return 16.0 * dofs + 24.0 * m.n_elems + 16.0 * pairs, flops


def work(case):
    """A solve or batch: the iterations it takes (about 20 for each factor of ten of the tolerance on these meshes)
    times one operator apply, one preconditioner apply and the vector updates; the preconditioner's least work is one
    read of r, one write of z and a conforming matrix of 3^d entries per row, in its own precision. The operands of a
    solve that stays in the card's caches are still counted once per iteration."""
    meshes = _batch_meshes(case) if case["kind"] == "batch" else [_mesh(case)]
    many = case.get("rhs", 1)
    total_b = total_f = 0.0
    for m in meshes:
        dofs = float(((m.p.astype(np.float64) + 1) ** m.dim).sum())
        ab, af = _apply_work(m)
        size = 8 if case.get("prec") == "fp64" else 4
        nnz = 0.6 * dofs * 3 ** m.dim
        pb, pf = 16.0 * dofs + nnz * (size + 4), 4.0 * nnz + 4.0 * dofs
        if case["kind"] == "apply":
            total_b, total_f = total_b + ab, total_f + af
        elif case["kind"] == "precond":
            total_b, total_f = total_b + pb, total_f + pf
        else:
            its = 20 * 10 if case.get("depth", 1) else 5 * 10
            total_b += many * its * (ab + pb + 48.0 * dofs)
            total_f += many * its * (af + pf + 10.0 * dofs)
    return {"bytes": total_b, "flops": total_f}


# ------------------------------------------------------------------ the same forms in 64 bits, by plain quadrature
def _gll(p):
    """The p + 1 Gauss-Lobatto points on [0, 1]."""
    inner = np.polynomial.legendre.Legendre.basis(p).deriv().roots() if p > 1 else np.zeros(0)
    return 0.5 * (np.concatenate([[-1.0], np.sort(inner.real), [1.0]]) + 1.0)


@functools.lru_cache(maxsize=None)
def _legendre_of_gll(p):
    L = np.polynomial.legendre
    inv = np.linalg.inv(L.legvander(2 * _gll(p) - 1, p))
    return inv, np.stack([2 * L.legder(np.eye(p + 1)[k], axis=0) for k in range(p + 1)], axis=1) @ inv


def _lagrange(p, t):
    """Values and derivatives of the degree-p Lagrange basis on the Gauss-Lobatto points at t, (len(t), p + 1)."""
    inv, der = _legendre_of_gll(p)
    v = np.polynomial.legendre.legvander(2 * np.asarray(t) - 1, p)
    return v @ inv, v[:, :len(der)] @ der


@functools.lru_cache(maxsize=None)
def _gauss(q):
    x, w = np.polynomial.legendre.leggauss(q)
    return 0.5 * (x + 1), 0.5 * w


def _kron(mats):
    """Tables per axis (x, y, ...) as one table, x fastest in rows and columns."""
    out = mats[0]
    for a in mats[1:]:
        out = (a[:, None, :, None] * out[None, :, None, :]).reshape(a.shape[0] * out.shape[0], -1)
    return out


def _points(axes):
    """The grid of per-axis points (x, y, ...), x fastest, (n, d)."""
    g = np.meshgrid(*reversed(axes), indexing="ij")
    return np.stack([a.ravel() for a in reversed(g)], axis=1)


def _corner_map(m):
    c, ext = np.asarray(m.corners).reshape(4, 2), np.asarray(m.extent, float) * m.lattice_h

    def at(X):
        s, t = X[..., 0:1] / ext[0], X[..., 1:2] / ext[1]
        x = (1 - s) * (1 - t) * c[0] + s * (1 - t) * c[1] + (1 - s) * t * c[2] + s * t * c[3]
        dx = ((1 - t) * (c[1] - c[0]) + t * (c[3] - c[2])) / ext[0]
        dy = ((1 - s) * (c[2] - c[0]) + s * (c[3] - c[1])) / ext[1]
        return x, np.stack([dx, dy], axis=-1)
    return at


def _geometry(m):
    """X -> (x, dx/dX) for the mesh's domain, or None for plain boxes."""
    if m.mapping is not None:
        def at(X):
            flat = X.reshape(-1, 2)
            return m.mapping(flat).reshape(X.shape), m.mapping.jacobian(flat).reshape(X.shape + (2,))
        return at
    return _corner_map(m) if m.corners is not None else None


def _touching(m):
    """(axis, left, right, lo, hi) per axis for each pair of touching elements once (right = -1, or left at an upper
    boundary with right = -1 and axis + d): the overlap in lattice units."""
    d, ext = m.dim, tuple(int(e) for e in m.extent)
    cells = np.full(tuple(e + 2 for e in ext), -1, dtype=np.int64)
    for s in np.unique(m.size):
        at = m.lo[m.size == s].astype(np.int64)
        ids = np.nonzero(m.size == s)[0]
        for off in np.ndindex(*([int(s)] * d)):
            cells[tuple((at + np.asarray(off) + 1).T)] = ids
    lo, hi = m.lo.astype(np.int64), m.lo.astype(np.int64) + m.size[:, None]
    for ax in range(d):
        a = np.take(cells, np.arange(ext[ax] + 1), axis=ax).ravel()
        b = np.take(cells, np.arange(1, ext[ax] + 2), axis=ax).ravel()
        for kind, keep in ((0, (a >= 0) & (b >= 0) & (a != b)), (1, (a >= 0) & (b < 0)), (2, (a < 0) & (b >= 0))):
            if not keep.any():
                continue
            pair = np.unique(np.stack([a[keep], b[keep]], axis=1), axis=0)
            if kind == 0:
                l, r = pair[:, 0], pair[:, 1]
                yield ax, l, r, np.maximum(lo[l], lo[r]), np.minimum(hi[l], hi[r])
            else:   # boundary: the element is `left`; its lower side goes by axis + d
                l = np.unique(pair[:, kind - 1])
                yield ax + (d if kind == 2 else 0), l, np.full(len(l), -1), lo[l], hi[l]


def _offsets(m):
    return np.concatenate([[0], np.cumsum((m.p.astype(np.int64) + 1) ** m.dim)])


def _load(m, seed):
    """int f phi_i for four random sine modes at the physical points, p + 3 Gauss points per direction."""
    r = inputs.sine_rhs(m.dim, seed)
    amps, waves = torch.from_numpy(r.amps).to(_device()), torch.from_numpy(r.waves.astype(float)).to(_device())
    geo, off, out = _geometry(m), _offsets(m), np.zeros(0)
    out = torch.zeros(int(off[-1]), dtype=torch.float64, device=_device())
    for p in np.unique(m.p):
        k = np.nonzero(m.p == p)[0]
        gx, gw = _gauss(int(p) + 3)
        phi = torch.from_numpy(_kron([_lagrange(int(p), gx)[0]] * m.dim)).to(_device())
        w = torch.from_numpy(_kron([gw[:, None]] * m.dim)[:, 0]).to(_device())
        h = m.size[k] * m.lattice_h
        X = (m.lo[k][:, None, :] * m.lattice_h + h[:, None, None] * _points([gx] * m.dim)[None])
        det = np.ones(X.shape[:2])
        if geo is not None:
            X, J = geo(X)
            det = np.linalg.det(J)
        X = torch.from_numpy(X).to(_device())
        f = sum(amps[i] * torch.sin(math.pi * waves[i] * X).prod(-1) for i in range(len(r.amps)))
        f = f * torch.from_numpy(det * (h ** m.dim)[:, None]).to(_device()) * w
        idx = torch.from_numpy(off[k][:, None] + np.arange(phi.shape[1])).to(_device())
        out[idx] = f @ phi
    return out


def _local(m, form, eta):
    """The form's local matrices: (DOF indices (g, n), matrices (g or 1, n, n)) for groups of elements and of
    touching pairs whose tables agree."""
    d, off, geo, dev = m.dim, _offsets(m), _geometry(m), _device()
    lh, coef = m.lattice_h, np.ones(m.n_elems) if m.coeff is None else np.asarray(m.coeff)
    up = lambda a: torch.from_numpy(np.array(a)).to(dev)  # noqa: E731
    h_el = m.size * lh
    h_pen = h_el.astype(float).copy()
    extra = 2 if geo is not None else 1
    dofs = lambda k: off[k][:, None] + np.arange((int(m.p[k[0]]) + 1) ** d)  # noqa: E731
    for p in np.unique(m.p):
        p = int(p)
        gx, gw = _gauss(p + extra)
        v, dv = _lagrange(p, gx)
        grad = np.stack([_kron([dv if a == i else v for a in range(d)]) for i in range(d)])
        w = _kron([gw[:, None]] * d)[:, 0]
        where = np.nonzero(m.p == p)[0]
        if geo is None:
            ref = up(np.einsum("iqm,q,iqn->mn", grad, w, grad, optimize=True))
            yield up(dofs(where)), up(coef[where] * h_el[where] ** (d - 2))[:, None, None] * ref
            continue
        for k in np.array_split(where, max(1, len(where) // 2000)):
            X = m.lo[k][:, None, :] * lh + h_el[k][:, None, None] * _points([gx] * d)[None]
            J = geo(X)[1]
            det = np.linalg.det(J)
            h_pen[k] = np.sqrt((det * w).sum(1)) * h_el[k]
            G = np.einsum("eqij,eqkj->eqik", np.linalg.inv(J), np.linalg.inv(J)) * (det * w * coef[k][:, None])[..., None, None]
            half = torch.einsum("eqij,jqn->eqin", up(G), up(grad))
            yield up(dofs(k)), torch.einsum("iqm,eqin->emn", up(grad), half)
    faces = list(_touching(m))
    if eta <= 0:
        count = np.zeros(m.n_elems, dtype=np.int64)
        for _, l, r, _, _ in faces:
            np.add.at(count, l, 1)
            np.add.at(count, r[r >= 0], 1)
        eta = 100.0 if form == "sipg" else float(count.max())
    for axis, left, right, lo, hi in faces:
        ax, sign, inside = axis % d, -1.0 if axis >= d else 1.0, right[0] >= 0
        tang = [t for t in range(d) if t != ax]
        rel = lambda k: [(lo[:, t] - m.lo[k, t]) for t in tang]  # noqa: E731
        key = [m.p[left], m.size[left], hi[:, tang[0]] - lo[:, tang[0]], *rel(left)]
        if inside:
            key += [m.p[right], m.size[right], *rel(right)]
        keys, which = np.unique(np.stack(key, axis=1), axis=0, return_inverse=True)
        order = np.argsort(which.ravel(), kind="stable")
        for part in np.split(order, np.cumsum(np.bincount(which.ravel()))[:-1]):
            l, r, f0 = left[part], right[part], part[0]
            sides = [(l, sign)] + ([(r, -1.0)] if inside else [])
            pe = max(int(m.p[k[0]]) for k, _ in sides)
            gx, gw = _gauss(pe + extra)
            length = float(hi[f0, tang[0]] - lo[f0, tang[0]])
            w = _kron([gw[:, None]] * (d - 1))[:, 0]
            vals, grads = [], []
            for k, sg in sides:
                p, s = int(m.p[k[0]]), float(m.size[k[0]])
                tabs = []
                for a in range(d):
                    t = (lo[f0, a] - m.lo[k[0], a] + length * gx) / s if a != ax else np.array([1.0 if sg > 0 else 0.0])
                    tabs.append(_lagrange(p, t))
                vals.append(_kron([tab[0] for tab in tabs]))
                grads.append(np.stack([_kron([tab[1] if a == i else tab[0] for a, tab in enumerate(tabs)])
                                       for i in range(d)]) / (s * lh))
            a = [coef[k] for k, _ in sides]
            amax = np.maximum(*a) if inside else a[0]
            share = 0.5 if inside else 1.0
            g = len(part)
            if geo is None:
                n = np.zeros((g, 1, d))
                n[..., ax] = sign
                ds = np.broadcast_to(w * (length * lh) ** (d - 1), (g, len(w)))
            else:
                X = np.empty((g, len(w), d))
                X[..., tang[0]] = (lo[part][:, tang[0]][:, None] + length * gx) * lh
                X[..., ax] = ((m.lo[l, ax] + (m.size[l] if sign > 0 else 0)) * lh)[:, None]
                J = geo(X)[1]
                Ji = np.linalg.inv(J)
                ds = w * length * lh * np.linalg.norm(J[..., tang[0]], axis=-1)
                n = sign * Ji[..., ax, :]
                n = n / np.linalg.norm(n, axis=-1, keepdims=True)
                n = np.einsum("gqij,gqj->gqi", Ji, n)   # the reference gradient's weight: J^-1 n
            same = geo is None and all(np.all(v == v[0]) for v in [*a, amax])   # one local matrix for the whole group
            if same:
                n, ds, amax, a = n[:1], ds[:1], amax[:1], [v[:1] for v in a]
            jump = up(np.concatenate([vals[0]] + ([-vals[1]] if inside else []), axis=1))
            flux = torch.cat([share * up(a[i])[:, None, None] * torch.einsum("gqi,iqn->gqn", up(np.broadcast_to(
                n, (n.shape[0], len(w), d))), up(grads[i])) for i in range(len(sides))], dim=2)
            wj = up(ds)[..., None] * jump
            mat = -torch.einsum("gqm,gqn->gmn", wj, flux)
            mat = mat + mat.transpose(1, 2)
            if form == "sipg":
                he = np.minimum(*[h_pen[k] for k, _ in sides]) if inside else h_pen[l]
                sigma = eta * pe * pe / he * (coef[l] if not inside else np.maximum(coef[l], coef[r]))
                sigma = sigma[:1] if same and np.all(sigma == sigma[0]) else sigma
                mat = up(sigma)[:, None, None] * torch.einsum("qm,gqn->gmn", jump, wj) + mat
            else:
                for i, (k, _) in enumerate(sides):
                    p = int(m.p[k[0]])
                    gv, gvw = _gauss(p + extra)
                    v1 = _lagrange(p, gv)[0]
                    if geo is None:
                        inv = _kron([np.linalg.inv(v1.T @ (gvw[:, None] * v1))] * d)
                        inv = up(inv / (h_el[k[0]] ** d))[None]
                    else:
                        X = m.lo[k][:, None, :] * lh + h_el[k][:, None, None] * _points([gv] * d)[None]
                        wv = np.linalg.det(geo(X)[1]) * _kron([gvw[:, None]] * d)[:, 0] * (h_el[k] ** d)[:, None]
                        vv = up(_kron([v1] * d))
                        inv = torch.linalg.inv(torch.einsum("qm,eq,qn->emn", vv, up(wv), vv))
                    lift = torch.einsum("qm,gqn->gmn", up(vals[i]), wj)
                    mat = mat + (eta * share * share * up(amax))[:, None, None] * (lift.transpose(1, 2) @ (inv @ lift))
            idx = np.concatenate([dofs(k) for k, _ in sides], axis=1)
            yield up(idx), mat


def _apply_exact(m, form, eta, x):
    y = torch.zeros_like(x)
    for idx, mat in _local(m, form, eta):
        y.index_add_(0, idx.reshape(-1), torch.einsum("gmn,gn->gm", mat.expand(len(idx), -1, -1), x[idx]).reshape(-1))
    return y


def _solve_exact(m, form, eta, loads):
    """x = A^-1 b for each load, by Jacobi-preconditioned CG on the assembled matrix."""
    n = loads.shape[0]
    rows, cols, vals = [], [], []
    for idx, mat in _local(m, form, eta):
        g, k = idx.shape
        rows.append(idx[:, :, None].expand(g, k, k).reshape(-1))
        cols.append(idx[:, None, :].expand(g, k, k).reshape(-1))
        vals.append(mat.expand(g, k, k).reshape(-1))
    A = torch.sparse_coo_tensor(torch.stack([torch.cat(rows), torch.cat(cols)]), torch.cat(vals), (n, n)).coalesce()
    at = A.indices()[0] == A.indices()[1]
    dinv = 1.0 / A.values()[at][:, None]
    A = A.to_sparse_csr()
    x, r = torch.zeros_like(loads), loads.clone()
    z = dinv * r
    p, rz = z.clone(), (r * z).sum(0)
    stop = 1e-14 * loads.norm(dim=0)
    for it in range(40000):
        q = A @ p
        alpha = rz / (p * q).sum(0).clamp_min(1e-300)
        x += alpha * p
        r -= alpha * q
        if it % 100 == 99 and bool((r.norm(dim=0) <= stop).all()):
            break
        z = dinv * r
        new = (r * z).sum(0)
        p = z + (new / rz.clamp_min(1e-300)) * p
        rz = new
    return x


def exact(case, seed):
    if case["kind"] == "precond":
        return None   # B holds the library's own multigrid hierarchy: nothing else defines its value
    if case["kind"] == "apply":
        m = _mesh(case)
        return _apply_exact(m, case["form"], case["eta"], _vector(_dofs([m])[0], seed))
    b = _loads(case, seed)
    if case["kind"] == "solve" and case["dim"] == 3 and len(b) > 20000:
        return None   # the assembled matrix alone takes longer than 20 s
    if case["kind"] == "solve":
        return _solve_exact(_mesh(case), case["form"], case["eta"], b[:, None])[:, 0]
    out, at = [], 0
    for m, n in zip(_batch_meshes(case), _dofs(_batch_meshes(case))):
        each = b[at:at + n * case["rhs"]].reshape(case["rhs"], n)
        at += n * case["rhs"]
        out.append(_solve_exact(m, "sipg", 0.0, each.t().contiguous()).t().reshape(-1))
    return torch.cat(out)
