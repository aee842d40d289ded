"""Which squares take the operator in Legendre modes (host rule, no GPU)."""
import numpy as np

from paper_2009_01287_gb300 import inputs


def _elems(p, n):
    e = np.zeros(9, dtype=np.int64)
    e[p] = n
    return e


def test_places_beyond_32_bits_stay_nodal(built_lib):
    """The records in modes hold places of traces in 32 bits; unknowns of degree 1
    have two places each, so a mesh the 32-bit unknowns admit (2^31 of them) can
    have more, and takes the nodal operator, which holds them in 64."""
    pays = built_lib.modal2_pays
    n = 1 << 28   # elements of degree 1: 2^30 unknowns
    assert pays(_elems(1, n - 1), 8 * (n - 1))
    assert not pays(_elems(1, n), 8 * n)
    assert not pays(_elems(1, 2 * n - 1), 8 * (2 * n - 1))


def test_br2_just_over_a_wave_stays_nodal(built_lib):
    """BR2 holds seven tiles on an SM: from 7.5 to 9 of them per SM the nodal
    operator is as fast or faster.  Degree 7: four elements to a tile."""
    pays = built_lib.modal2_pays
    for per_sm, br2 in [(5.9, False), (6, True), (7.49, True), (7.5, False), (8, False), (8.99, False), (9, True),
                        (20, True)]:
        elems = _elems(7, 4 * int(np.ceil(per_sm * 152)))
        assert pays(elems, 10 ** 6, br2=True) == br2, per_sm
        assert pays(elems, 10 ** 6, br2=False) == (per_sm >= 6)


def test_places_of_a_mesh(built_lib):
    """A square of edge 4 and degree 3 beside sixteen unit squares of degree 1:
    the sides' traces, and those of the large one restricted to four sub-faces."""
    lo = [(0, 0)] + [(4 + i % 4, i // 4) for i in range(16)]
    mesh = inputs.MeshDesc(dim=2, lo=np.array(lo, dtype=np.int32), size=np.array([4] + [1] * 16, dtype=np.int32),
                           p=np.array([3] + [1] * 16, dtype=np.int32), extent=(8, 4), lattice_h=0.125)
    hs = built_lib.HostSetup(mesh, built_lib.make_options(), amg=False)
    assert hs.modal2_places() == 4 * 4 + 16 * 4 * 2 + 4 * 4


def test_items_of_a_mesh_in_modes(built_lib):
    """The nodal kernel's item lists, formed for inspection only where the
    operator takes modes: every sub-face once."""
    n = 912 * 3 + 1   # a strip of degree 8, three elements to a tile
    mesh = inputs.MeshDesc(dim=2, lo=np.stack([np.arange(n), np.zeros(n)], axis=1).astype(np.int32),
                           size=np.ones(n, dtype=np.int32), p=np.full(n, 8, dtype=np.int32), extent=(n, 1),
                           lattice_h=1.0 / n)
    hs = built_lib.HostSetup(mesh, built_lib.make_options(), amg=False)
    assert built_lib.modal2_pays(_elems(8, n), hs.modal2_places())
    ptr, items, chunk, info = hs.face_items()
    assert np.array_equal(np.sort(items[:, 0]), np.arange(4 * n))
    assert np.array_equal(np.diff(ptr), chunk) and ptr[-1] == 4 * n
    assert int((info[:, 0] == 1).sum()) == 2 * (n - 1)
