"""Group ranges of the CUDA-core mass pass (csrc/group_ranges.h): over shapes and
SM counts, the ranges take every group exactly once, in order, and the anchor
(group G) once, in the last range."""
import itertools

from tests.group_ranges import ranges


def test_every_group_once_and_the_anchor_once():
    calls = [(G, RG, ar, keyu, nsm) for G, RG, (ar, keyu), nsm in itertools.product(
        (0, 1, 2, 3, 5, 8, 9, 10, 31, 32, 97, 1024), (16, 48, 112, 512),
        ((16, 1), (16, 8), (32, 128), (16, 256), (16, 3000), (64, 100000)), (1, 76, 148, 152, 160))]
    owns = 0
    for (G, *_), (gper, own, rs) in zip(calls, ranges(calls)):
        taken = [g for g0, g1 in rs for g in range(g0, g1)]
        assert taken == list(range(G + 1)), (G, gper, own, rs)
        assert all(g1 > g0 for g0, g1 in rs)
        assert own == (rs[-1] == (G, G + 1) and G > 0), (G, gper, own, rs)
        assert all(g1 - g0 == gper for g0, g1 in rs[:-2])
        owns += own
    assert 0 < owns < len(calls)
