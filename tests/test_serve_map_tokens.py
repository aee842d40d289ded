"""The served form's numbers of map objects (host logic, no GPU): one of its own
per object whether it takes weak references or not, and no more than a bounded
number of the latter kept alive."""
import gc
import sys

from paper_2009_01287_gb300 import inputs, serve


class Slotted:
    """A map that takes no weak reference."""
    __slots__ = ()

    def __call__(self, x):
        return x


def test_tokens_are_the_objects_own():
    for make in (inputs.WavyMap, Slotted):
        maps = [make() for _ in range(20)]
        tokens = [serve._map_token(f) for f in maps]
        assert len(set(tokens)) == 20
        assert [serve._map_token(f) for f in maps] == tokens
        del maps
        gc.collect()
        again = [make() for _ in range(20)]   # may take the ids of the first ones
        assert not set(tokens) & {serve._map_token(f) for f in again}


def test_objects_without_weak_references_are_given_back():
    f = Slotted()
    alone = sys.getrefcount(f)
    first = serve._map_token(f)
    assert sys.getrefcount(f) > alone
    others = [Slotted() for _ in range(500)]
    assert len({serve._map_token(g) for g in others} | {first}) == 501
    assert sys.getrefcount(f) == alone               # no longer kept
    assert len(serve._map_kept) <= serve._MAP_KEPT
    assert serve._map_token(f) > first               # a new number, not another's
