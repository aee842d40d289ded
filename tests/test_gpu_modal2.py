"""The operator of squares in Legendre modes at the edges of its tile lists:
sides with more sub-faces than one round of a warp's work space takes,
neighbours of the lowest and of higher degrees on them, sub-faces four levels
below their neighbour, tiles of one element and full ones of every degree, a
hole and a jumping coefficient, on meshes just large enough to take it.  Sampled
rows against the FP64 oracle to 1e-12 relative, the bound of every operator test here (FP64 sums of at most a few hundred terms:
about 1e-14)."""
import numpy as np
import pytest

from oracle import dg
from oracle.topology import Topology
from paper_2009_01287_gb300 import inputs

pytestmark = pytest.mark.gpu


def _mesh(lo, size, p, extent):
    return inputs.MeshDesc(dim=2, lo=np.array(lo, dtype=np.int32), size=np.array(size, dtype=np.int32),
                           p=np.array(p, dtype=np.int32), extent=extent, lattice_h=1.0 / extent[0])


def _between_small(pbig, psmall, n=16):
    """A square of edge n with two columns of n unit squares on either side of it."""
    lo, size, p = [(n, 0)], [n], [pbig]
    for x0 in (0, 2 * n):
        for y in range(n):
            for x in range(n):
                lo.append((x0 + x, y))
                size.append(1)
                p.append(psmall)
    return _mesh(lo, size, p, (3 * n, n))


def _corner_chain(pbig, psmall):
    """Four cells, one of them split towards the domain's centre four times."""
    lo, size, p = [], [], []
    for c in range(1, 4):
        lo.append((16 * (c & 1), 16 * (c >> 1)))
        size.append(16)
        p.append(pbig)
    at, s = 0, 16
    while s > 1:
        s //= 2
        for c in range(4 if s == 1 else 3):
            lo.append((at + s * (c & 1), at + s * (c >> 1)))
            size.append(s)
            p.append(psmall)
        at += s
    return _mesh(lo, size, p, (32, 32))


def _stack(mesh, copies):
    """Copies of a mesh on top of each other."""
    lo = np.asarray(mesh.lo).reshape(-1, 2)
    up = np.array([0, mesh.extent[1]], dtype=np.int32)
    return _mesh(np.concatenate([lo + k * up for k in range(copies)]), np.tile(mesh.size, copies),
                 np.tile(mesh.p, copies), (mesh.extent[0], mesh.extent[1] * copies))


def _apply(B, device, mesh, form):
    """(x, y = A x, eta) through the kernels in modes."""
    import torch
    tiles = sum(-(-int((np.asarray(mesh.p) == p).sum()) // (32 // (p + 1))) for p in range(1, 9))
    assert tiles >= 6 * 152   # the size from which the operator takes modes
    eta = dg.br2_eta(Topology(mesh.lo, mesh.size, mesh.p, mesh.extent)) if form == "br2" else 100.0
    M = B.Mesh(mesh, B.make_options(form=B.DG_FORM_BR2 if form == "br2" else B.DG_FORM_SIPG, eta=eta))
    x = inputs.random_vector(M.n_dofs, 9)
    xd = torch.tensor(x, dtype=torch.float64, device=device)
    yd = torch.full_like(xd, float("nan"))
    B.dg_apply(M.h, xd, yd)
    torch.cuda.synchronize()
    y = yd.cpu().numpy()
    assert np.isfinite(y).all()
    return x, y, eta


def _compare(pairs):
    scale = max(np.abs(r).max() for _, r in pairs)
    for y, r in pairs:
        assert np.abs(y - r).max() <= 1e-12 * scale


def _check_stack(B, device, unit, copies, form, elems):
    """Elements (copy, element of the unit) of a stack.  Their rows come from the
    oracle on the copy and the ones below and above it, moved to the origin: at
    a height of hundreds of lattice cells the oracle's coordinates lose the
    digits that the bound asks for (2e-12 between two of its quadratures)."""
    x, y, eta = _apply(B, device, _stack(unit, copies), form)
    n = len(unit.p)
    dofs = int(((np.asarray(unit.p, dtype=np.int64) + 1) ** 2).sum())
    spaces, pairs = {}, []
    for c, k in elems:
        lo, hi = max(0, c - 1), min(copies, c + 2)
        if hi - lo not in spaces:
            m = _stack(unit, hi - lo)
            spaces[hi - lo] = dg.DGSpace(Topology(m.lo, m.size, m.p, m.extent), unit.lattice_h)
        space = spaces[hi - lo]
        at, e = lo * dofs, (c - lo) * n + k
        pairs.append((y[at + space.dofs(e)], dg.element_rows(space, e, x[at:hi * dofs], eta, form)))
    _compare(pairs)


@pytest.mark.parametrize("form", ["sipg", "br2"])
@pytest.mark.parametrize("mesh,copies", [(_between_small(8, 1), 30), (_between_small(2, 3), 16),
                                         (_between_small(1, 8, 4), 85), (_corner_chain(5, 2), 520),
                                         (_corner_chain(1, 4), 500)],
                         ids=["rounds", "higher-small", "highest-small", "deep", "deep-low"])
def test_modal_operator_at_hanging_sides(built_lib, cuda_device, mesh, copies, form):
    n = len(mesh.p)
    elems = [(0, k) for k in range(0, n, max(1, n // 20))] + [(copies // 2, k) for k in range(4)] + [(copies - 1, 0)]
    _check_stack(built_lib, cuda_device, mesh, copies, form, elems)


@pytest.mark.parametrize("form", ["sipg", "br2"])
@pytest.mark.parametrize("p", range(1, 9))
def test_modal_operator_of_one_degree(built_lib, cuda_device, p, form):
    """Full tiles and a remainder of one element (a 1 x n strip)."""
    n = 912 * (32 // (p + 1)) + 1
    unit = _mesh([(0, 0)], [1], [p], (1, 1))
    _check_stack(built_lib, cuda_device, unit, n, form, [(c, 0) for c in (0, 1, n // 2, n - 2, n - 1)])


@pytest.mark.parametrize("form", ["sipg", "br2"])
def test_modal_operator_holes_and_coefficient(built_lib, cuda_device, form):
    """Whole vectors against the library's host operator (checked against the
    oracle on small meshes): on these lattices, 320 and 384 cells across, two
    quadratures of the oracle differ by 1e-12 themselves."""
    B = built_lib
    coef = inputs.random_refined_mesh(2, 40, 3, 0.3, 1, 8, 5)
    for mesh in (inputs.lshape(inputs.random_refined_mesh(2, 48, 3, 0.3, 1, 8, 3)),
                 inputs.with_coeff(coef, inputs.base_parity_coeff(coef, 40))):
        x, y, eta = _apply(B, cuda_device, mesh, form)
        host = B.HostSetup(mesh, B.make_options(form=B.DG_FORM_BR2 if form == "br2" else B.DG_FORM_SIPG, eta=eta),
                           amg=False)
        _compare([(y, host.apply(x))])
