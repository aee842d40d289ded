"""Host planning of the cubes' hanging sub-faces (no GPU): a side may have any
number of them (65,536 and one more unit cubes on a side of edge 256: one tile
then holds more sub-faces than 16 bits count), every sub-face between a larger
and a smaller side is one pair, and the results of a side's pairs lie one after
another where the side reads them."""
import numpy as np
import pytest

from paper_2009_01287_gb300 import inputs


def beside(n, pbig, psmall):
    """A cube of edge n, a layer of n x n unit cubes on its upper x side."""
    y, z = np.meshgrid(np.arange(n), np.arange(n))
    lo = np.stack([np.full(n * n, n), y.ravel(), z.ravel()], axis=1)
    return inputs.MeshDesc(dim=3, lo=np.concatenate([[[0, 0, 0]], lo]).astype(np.int32),
                           size=np.concatenate([[n], np.ones(n * n)]).astype(np.int32),
                           p=np.array([pbig] + [psmall] * (n * n), dtype=np.int32), extent=(n + 1, n, n),
                           lattice_h=1.0 / n)


def _check(B, mesh, form):
    hs = B.HostSetup(mesh, B.make_options(form=B.DG_FORM_BR2 if form == "br2" else B.DG_FORM_SIPG), amg=False)
    pairs, sides = hs.hanging3()
    big, small = mesh.size.max(), mesh.size.min()
    assert len(sides) == 6 * mesh.n_elems and big > small
    # places of the elements' traces, then of the results
    n2 = (mesh.p.astype(np.int64) + 1) ** 2
    end = 6 * int(n2.sum())
    assert (pairs[:, :2] >= 0).all() and (pairs[:, :2] < end).all()
    starts = np.concatenate([pairs[:, 2], pairs[:, 3]])
    width = np.concatenate([pairs[:, 4], pairs[:, 5]])
    order = np.argsort(starts)
    assert starts[order][0] == end                              # results fill their part without gaps or overlaps
    assert np.array_equal(starts[order] + width[order], np.append(starts[order][1:], end + width.sum()))
    # the sides read all of them, each once
    hang = sides[sides[:, 2] > 0]
    read = np.concatenate([f + n2[k] * np.arange(c) for k, f, c in hang])
    assert np.array_equal(np.sort(read), starts[order])
    return len(pairs), int(sides[:, 2].max())


@pytest.mark.parametrize("form", ["sipg", "br2"])
def test_every_pair_once(built_lib, form):
    for seed in (1, 2):
        mesh = inputs.small_hp_mesh(seed, base=3, depth=2, prob=0.3, pmax=4, dim=3)
        assert _check(built_lib, mesh, form)[0] > 0
    assert _check(built_lib, beside(4, 3, 1), form) == (16, 16)


def test_side_of_many_sub_faces(built_lib):
    assert _check(built_lib, beside(256, 1, 1), "sipg") == (65536, 65536)


def test_places_beyond_32_bits(built_lib):
    """Cubes of degree 1 have three places of traces per unknown, so a mesh the
    32-bit unknowns admit can need 64-bit places."""
    mesh = inputs.small_hp_mesh(1, base=3, depth=2, prob=0.3, pmax=4, dim=3)
    hs = built_lib.HostSetup(mesh, built_lib.make_options(), amg=False)
    pairs, sides = hs.hanging3()
    first = 3 * (1 << 31)
    far, far_sides = hs.hanging3(first)
    assert np.array_equal(far[:, :4], pairs[:, :4] + first) and np.array_equal(far[:, 4:], pairs[:, 4:])
    assert np.array_equal(far_sides[:, 1], sides[:, 1] + first)
    assert np.array_equal(far_sides[:, [0, 2]], sides[:, [0, 2]])
