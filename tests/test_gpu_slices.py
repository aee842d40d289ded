"""The preconditioner's sparse rows at the edges of their slices: a cube mesh
whose coarse corner touches three faces of many small elements, so that rows of
P^T and of the low-order matrix range from one entry to several thousand (one
lane, a warp, a whole CTA per row), and meshes so small that most slices are
partly empty.  FP64, against the oracle to 1e-12 of the largest entry, the
bound of every preconditioner test here."""
import numpy as np
import pytest

from oracle import solver
from paper_2009_01287_gb300 import inputs

pytestmark = pytest.mark.gpu


def _corner(psmall, split=2):
    """Eight cells of edge 2^split; the three face neighbours of the first are grids of unit cubes."""
    s = 1 << split
    lo, size, p = [], [], []
    for c in range(8):
        o = [s * ((c >> d) & 1) for d in range(3)]
        if c in (1, 2, 4):
            for i in range(s ** 3):
                lo.append((o[0] + i % s, o[1] + i // s % s, o[2] + i // s ** 2))
                size.append(1)
                p.append(psmall)
        else:
            lo.append(tuple(o))
            size.append(s)
            p.append(1)
    return inputs.MeshDesc(dim=3, lo=np.array(lo, dtype=np.int32), size=np.array(size, dtype=np.int32),
                           p=np.array(p, dtype=np.int32), extent=(2 * s,) * 3, lattice_h=0.5 / s)


MESHES = {
    "long-rows": (lambda: _corner(3), "br2"),
    "warp-rows": (lambda: _corner(2), "sipg"),
    "tiny-2d": (lambda: inputs.uniform_mesh(2, 2, 1), "sipg"),
    "small-2d": (lambda: inputs.small_hp_mesh(5, base=3, depth=3, prob=0.5, pmin=1, pmax=8), "sipg"),
}


@pytest.mark.parametrize("name", list(MESHES))
def test_precond_rows_of_every_length(built_lib, cuda_device, name):
    import torch
    B = built_lib
    mk, form = MESHES[name]
    mesh = mk()
    prob = solver.build_problem(mesh, form=form)
    ref = solver.Preconditioner(prob, lor="amg").apply
    M = B.Mesh(mesh, B.make_options(form=B.DG_FORM_BR2 if form == "br2" else B.DG_FORM_SIPG))
    pc = B.Precond(M)
    r = inputs.random_vector(M.n_dofs, 11)
    rd = torch.tensor(r, dtype=torch.float64, device=cuda_device)
    zd = torch.full_like(rd, float("nan"))
    B.dg_precond_apply(pc.h, rd, zd)
    torch.cuda.synchronize()
    z = ref(r)
    assert np.abs(zd.cpu().numpy() - z).max() <= 1e-12 * np.abs(z).max()
