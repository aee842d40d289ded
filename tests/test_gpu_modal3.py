"""The cube operator in Legendre modes at the edges of its tile lists: a large
element of the highest degree whose hanging sub-faces need more than one round
of the tile's scratch, neighbours of the lowest and of higher degrees on them,
and a sub-face four levels below its neighbour (uneven positions of the
restriction).  Against the FP64 oracle to 1e-12 relative, the bound of every
operator test here (FP64 sums of at most a few hundred terms: about 1e-14)."""
import numpy as np
import pytest

from oracle import solver
from paper_2009_01287_gb300 import inputs

pytestmark = pytest.mark.gpu


def _between_small(pbig, psmall):
    """A cube of edge 4 with a 4x4x4 grid of unit cubes on either side."""
    lo, size, p = [(4, 0, 0)], [4], [pbig]
    for x0 in (0, 8):
        for z in range(4):
            for y in range(4):
                for x in range(4):
                    lo.append((x0 + x, y, z))
                    size.append(1)
                    p.append(psmall)
    return inputs.MeshDesc(dim=3, lo=np.array(lo, dtype=np.int32), size=np.array(size, dtype=np.int32),
                           p=np.array(p, dtype=np.int32), extent=(12, 4, 4), lattice_h=1.0 / 12)


def _corner_chain(pbig, psmall):
    """Eight cells, one of them split towards the domain's centre four times."""
    lo, size, p = [], [], []
    for c in range(1, 8):
        lo.append(tuple(16 * ((c >> d) & 1) for d in range(3)))
        size.append(16)
        p.append(pbig)
    at, s = 0, 16
    while s > 1:
        s //= 2
        for c in range(8 if s == 1 else 7):
            lo.append(tuple(at + s * ((c >> d) & 1) for d in range(3)))
            size.append(s)
            p.append(psmall)
        at += s
    return inputs.MeshDesc(dim=3, lo=np.array(lo, dtype=np.int32), size=np.array(size, dtype=np.int32),
                           p=np.array(p, dtype=np.int32), extent=(32, 32, 32), lattice_h=1.0 / 32)


@pytest.mark.parametrize("form", ["sipg", "br2"])
@pytest.mark.parametrize("mesh", [_between_small(8, 1), _between_small(2, 3), _corner_chain(5, 2), _corner_chain(1, 4)],
                         ids=["rounds", "higher-small", "deep", "deep-low"])
def test_modal_operator_at_hanging_faces(built_lib, cuda_device, mesh, form):
    import torch
    B = built_lib
    _, _, A = solver.build_operator(mesh, form=form)
    M = B.Mesh(mesh, B.make_options(form=B.DG_FORM_BR2 if form == "br2" else B.DG_FORM_SIPG))
    x = inputs.random_vector(M.n_dofs, 9)
    xd = torch.tensor(x, dtype=torch.float64, device=cuda_device)
    yd = torch.full_like(xd, float("nan"))
    B.dg_apply(M.h, xd, yd)
    torch.cuda.synchronize()
    ref = A @ x
    assert np.abs(yd.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
