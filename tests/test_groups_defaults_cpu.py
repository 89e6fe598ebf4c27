"""The built-in tile table of the grouped Gram given by value (DEFAULT_TILES) and left out are one plan: a
workspace prepared with the one is used with the other, on both sides of the object count at which
the defaults grow. Host planning only; the plan's lists show in the workspace size."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def t3f():
    from paper_1801_01928_gb300 import build
    path = build.build()
    import paper_1801_01928_gb300 as t3f
    t3f.load(path)
    return t3f


@pytest.mark.parametrize("count", [12, 255, 256, 300, 512])
def test_default_table_by_value_is_the_default(t3f, count):
    torch = pytest.importorskip("torch")
    b = t3f._binding
    ranks = [[1, 2 + o % 40, 2 + o % 40, 1] for o in range(count)]
    sizes = [t3f.RaggedTT.object_numel([2, 2, 2], r) for r in ranks]
    X = t3f.RaggedTT(torch.empty(sum(sizes)), [3] * count, [[2, 2, 2]] * count, ranks,
                     [sum(sizes[:o]) for o in range(count)])

    def size(tiles):
        return t3f.load().t3f_gram_groups_workspace_size(ctypes.byref(X.desc()), 1, b._i32([0, count]), b._tiles_arg(tiles))

    assert size(None) == size(t3f.DEFAULT_TILES) > 0
    assert size((10, 6, 3, 0)) == 0 and size((17, 6, 3, 1)) == 0
