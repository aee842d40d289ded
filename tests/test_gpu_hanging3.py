"""The cube operator where one side has more sub-faces than 16 bits count: a
cube of edge 256 against a layer of unit cubes.  The whole vector against the
library's host operator (checked against the oracle on small meshes) to 1e-12
relative: a residual of the large cube sums 65,536 terms of either sign in one
order, whose rounding is some 256 units of its last place, 3e-14."""
import numpy as np
import pytest

from test_host_hanging3 import beside

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["sipg", "br2"])
def test_operator_on_a_side_of_many_sub_faces(built_lib, cuda_device, form):
    import torch
    from paper_2009_01287_gb300 import inputs
    B = built_lib
    mesh = beside(256, 1, 1)
    opts = B.make_options(form=B.DG_FORM_BR2 if form == "br2" else B.DG_FORM_SIPG, eta=100.0)
    M = B.Mesh(mesh, opts)
    x = inputs.random_vector(M.n_dofs, 3)
    xd = torch.tensor(x, dtype=torch.float64, device=cuda_device)
    yd = torch.full_like(xd, float("nan"))
    B.dg_apply(M.h, xd, yd)
    torch.cuda.synchronize()
    ref = B.HostSetup(mesh, opts, amg=False).apply(x)
    assert np.abs(yd.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
