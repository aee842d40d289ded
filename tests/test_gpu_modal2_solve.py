"""Squares in Legendre modes beyond the stand-alone apply: inside a solve (p
formed in the modes' kernel, p . q, the step, the stop), without allocation, in
a batch whose members are nodal by themselves, and with tuned tiles.

True residuals come from the library's host operator (checked against the oracle
on small meshes): the solver's own, updated by recurrence in FP64, differs from
it by rounding times the condition number, up to 1e5 on these meshes: 1e-11, a
hundredth of the tightest tolerance here.  Two solutions of relative residual
1e-9 differ by at most the condition number times 2e-9, 2e-4."""
import numpy as np
import pytest

from paper_2009_01287_gb300 import inputs

pytestmark = pytest.mark.gpu


def _in_modes(B, meshes, n_rhs=1, br2=False):
    elems = sum(np.bincount(np.asarray(m.p), minlength=9) for m in meshes) * n_rhs
    return B.modal2_pays(elems, 0, br2)


def _options(B, form, **kw):
    return B.make_options(form=B.DG_FORM_BR2 if form == "br2" else B.DG_FORM_SIPG,
                          eta=40.0 if form == "br2" else 100.0, **kw)


def _residual(host, b, x):
    b, x = b.cpu().numpy(), x.cpu().numpy()
    return np.linalg.norm(b - host.apply(x)) / np.linalg.norm(b)


@pytest.mark.parametrize("form", ["sipg", "br2"])
def test_solve_in_modes(built_lib, cuda_device, form, monkeypatch):
    import torch
    B = built_lib
    mesh = inputs.random_refined_mesh(2, 48, 3, 0.3, 1, 3, 5)
    assert _in_modes(B, [mesh], br2=form == "br2")
    opts = _options(B, form)
    M = B.Mesh(mesh, opts)
    graph = B.Precond(M, opts)
    monkeypatch.setenv("DG_PCG_GRAPH", "0")
    loop = B.Precond(M, opts)
    host = B.HostSetup(mesh, opts, amg=False)
    b = torch.tensor(inputs.random_vector(M.n_dofs, 7), dtype=torch.float64, device=cuda_device)
    for rtol, maxit in [(1e-8, 2000)] + [(1e-12, m) for m in (1, 2, 3, 4, 6, 7, 9)]:
        x = {}
        for name, pc in (("graph", graph), ("loop", loop)):
            x[name] = torch.full_like(b, 3.0)
            i = B.dg_pcg_solve(M.h, pc.h, b, x[name], rtol, maxit, raise_on_notconv=False)
            x[name, "info"] = (i.iters, i.status, i.rel_res)
        assert x["graph", "info"] == x["loop", "info"]
        assert torch.equal(x["graph"], x["loop"])
        iters, status, rel = x["graph", "info"]
        true = _residual(host, b, x["graph"])
        if maxit == 2000:
            assert status == B.DG_OK and true <= 1.01e-8
            y = torch.full_like(b, 3.0)
            j = B.dg_pcg_solve_noalloc(M.h, graph.h, b, y, rtol, maxit)
            assert j.iters == iters and torch.equal(x["graph"], y)
        else:
            assert iters == maxit
        assert abs(true - rel) <= 0.01 * rel
    x0 = torch.full_like(b, 3.0)
    i = B.dg_pcg_solve(M.h, graph.h, torch.zeros_like(b), x0, 1e-8, 50)
    assert i.iters == 0 and not x0.any()


@pytest.mark.parametrize("form", ["sipg", "br2"])
def test_batch_in_modes_of_nodal_members(built_lib, cuda_device, form):
    """Members of different size, degree and hanging levels, one with a jumping
    coefficient; three loads each, one of them zero, so that instances stop at
    different iterations and their tiles idle while others go on."""
    import torch
    B = built_lib
    meshes = [inputs.random_refined_mesh(2, 5 + 2 * k, 3, 0.35, 1, 2 + k % 5, 20 + k) for k in range(9)]
    meshes[3] = inputs.with_coeff(meshes[3], inputs.base_parity_coeff(meshes[3], 11))
    meshes.append(inputs.uniform_mesh(2, 3, 8))
    br2 = form == "br2"
    assert _in_modes(B, meshes, 3, br2) and not any(_in_modes(B, [m], br2=br2) for m in meshes)
    opts = _options(B, form, precision=B.DG_PREC_FP64)
    bat = B.Batch(meshes, n_rhs=3, opts=opts)
    b = torch.tensor(inputs.random_vector(bat.n_dofs, 3), dtype=torch.float64, device=cuda_device)
    zero = 4 * 3 + 1
    b[bat.offsets[zero]:bat.offsets[zero + 1]] = 0.0
    x = torch.full_like(b, 5.0)
    res, _ = bat.solve(b, x, 1e-9, 3000)
    counts = set()
    for k, m in enumerate(meshes):
        M = B.Mesh(m, opts)
        pc = B.Precond(M, opts)
        host = B.HostSetup(m, opts, amg=False)
        for r in range(3):
            i = 3 * k + r
            seg, xi = b[bat.offsets[i]:bat.offsets[i + 1]], x[bat.offsets[i]:bat.offsets[i + 1]]
            if i == zero:
                assert res[i].iters == 0 and not xi.any()
                continue
            x1 = torch.empty_like(seg)
            info = B.dg_pcg_solve(M.h, pc.h, seg.clone(), x1, 1e-9, 3000)
            assert res[i].status == B.DG_OK and abs(res[i].iters - info.iters) <= 1
            assert _residual(host, seg, xi) <= 1.01e-9
            assert float((xi - x1).abs().max()) <= 2e-4 * float(x1.abs().max())
            counts.add(res[i].iters)
    assert len(counts) > 5


@pytest.mark.parametrize("form", ["sipg", "br2"])
def test_tuned_tiles_in_modes(built_lib, cuda_device, form):
    """Other tiles, the same sums: y = A x to a few units of rounding, and a solve."""
    import torch
    B = built_lib
    mesh = inputs.random_refined_mesh(2, 50, 3, 0.3, 1, 3, 5)
    assert _in_modes(B, [mesh], br2=form == "br2")
    M = B.Mesh(mesh, _options(B, form))
    T = B.Mesh(mesh, _options(B, form, tune_tiles=1))
    assert T.stats.tiles_tuned == 1
    assert all(1 <= T.stats.tile_elems[p] <= 32 // (p + 1) for p in (1, 2, 3))
    x = torch.tensor(inputs.random_vector(M.n_dofs, 2), dtype=torch.float64, device=cuda_device)
    y, z = torch.empty_like(x), torch.empty_like(x)
    B.dg_apply(M.h, x, y)
    B.dg_apply(T.h, x, z)
    torch.cuda.synchronize()
    assert float((y - z).abs().max()) <= 1e-14 * float(y.abs().max())
    pc = B.Precond(T)
    u = torch.empty_like(x)
    assert B.dg_pcg_solve(T.h, pc.h, x, u, 1e-8, 2000).status == B.DG_OK
    host = B.HostSetup(mesh, _options(B, form), amg=False)
    assert _residual(host, x, u) <= 1.01e-8


@pytest.mark.parametrize("base,pmax,coef", [(44, 8, True), (56, 4, False)], ids=["coefficient", "holes"])
def test_br2_apply_over_a_wave(built_lib, cuda_device, base, pmax, coef):
    """BR2 above the tiles per SM at which it stays nodal, to 1e-12 of the host
    operator, the bound of every operator test here."""
    import torch
    B = built_lib
    mesh = inputs.random_refined_mesh(2, base, 3, 0.3, 1, pmax, 5)
    mesh = inputs.with_coeff(mesh, inputs.base_parity_coeff(mesh, base)) if coef else mesh
    if not coef:
        mesh = inputs.lshape(inputs.random_refined_mesh(2, 64, 3, 0.3, 1, pmax, 5))
    assert _in_modes(B, [mesh], br2=True)
    opts = _options(B, "br2")
    M = B.Mesh(mesh, opts)
    x = inputs.random_vector(M.n_dofs, 4)
    xd = torch.tensor(x, dtype=torch.float64, device=cuda_device)
    yd = torch.full_like(xd, float("nan"))
    B.dg_apply(M.h, xd, yd)
    torch.cuda.synchronize()
    ref = B.HostSetup(mesh, opts, amg=False).apply(x)
    assert np.abs(yd.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
