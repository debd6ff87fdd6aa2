"""Placement sorts its candidates by their 32-bit keys alone and puts equal keys
into voxel order afterwards: from one molecule to a full lattice (keys of 22 to
32 bits; 500,000 voxels hold about 30 pairs of equal keys), compared voxel by
voxel with the oracle's order."""
import numpy as np
import pytest

from test_gpu_parity import build_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts", [(1, 0), (500, 3), (200000, 60001), (250000, 249999), (500000, 0)])
def test_placement_order(counts):
    def recipe(L):
        for n in counts:
            L.add_species(1e-12, n)
    g, o = build_both((100, 100, 50), recipe, 29)
    assert np.array_equal(np.asarray(g.grid()).ravel(), np.asarray(o.grid()).ravel())
    for s in range(len(counts)):
        a, b = g.coords(s), o.coords(s)
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
