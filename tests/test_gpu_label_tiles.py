"""Tiled labelling at its edges against the oracle's full scan: ragged tiles, more generators
near a tile than its list holds, a single generator, and exact ties (coincident generators,
generators on a lattice whose bisecting planes pass through voxel centres)."""
import numpy as np
import pytest

from oracle.voronoi import label_rve

pytestmark = pytest.mark.gpu


def _lattice(n):
    g = (np.arange(n) + 0.25) / n
    return np.stack(np.meshgrid(g, g, g, indexing="ij"), axis=-1).reshape(-1, 3)


@pytest.mark.parametrize("shape,n,seeds", [
    ((9, 17, 33), 700, "random"), ((4, 4, 4), 2000, "random"), ((5, 9, 20), 1, "random"),
    ((1, 30, 50), 40, "random"), ((40, 1, 1), 7, "random"), ((64, 64, 64), 30, "random"),
    ((16, 16, 16), 64, "lattice"), ((24, 24, 24), 40, "coincident"),
])
def test_tiled_labels_equal_full_scan(lib, cuda, shape, n, seeds):
    from paper_2402_09996_gb300 import inputs, rve

    inp = inputs.make_inputs(shape, n, 0.5, 11)
    if seeds == "lattice":
        inp.seeds[:] = _lattice(4)
    elif seeds == "coincident":
        inp.seeds[n // 2:] = inp.seeds[: n - n // 2]
    got = rve.label_voronoi(inp)
    assert np.array_equal(got.astype(np.int64), label_rve(inp))
