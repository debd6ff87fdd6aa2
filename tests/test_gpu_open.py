"""Claim and commit launches that skip the claims of hops no other molecule can
contest, bit for bit against the oracle.

They take lists of 262,144 molecules and more; here on lattices where the
test of the twelve neighbours can go wrong: bricks that line up across a
periodic wrap and bricks that do not, walls, partial bricks, FCC layers, an odd
number of layers, compartments, both kinds of claims, few and many neighbours.
"""
import numpy as np
import pytest

import models
import paper_1605_03726_gb300 as psc
from test_gpu_parity import assert_same, build_both

pytestmark = pytest.mark.gpu

N = 1 << 18

CASES = [
    ("bricks", (128, 128, 96), 7, N),
    ("dense", (96, 80, 64), 7, N + 100000),
    ("walls", (131, 127, 93), 0, N),
    ("partial_i", (126, 120, 90), 7, N),                        # ni and nj not multiples of 4 across the wrap
    ("partial_mixed", (129, 118, 91), psc.PERIODIC_I, N + 1),
    ("sparse", (160, 160, 150), 7, N),
    ("fcc", (120, 112, 96), 7 | psc.FCC, N),
    ("fcc_odd_layers", (120, 112, 93), 7 | psc.FCC, N),
    ("fcc_walls", (117, 110, 95), psc.FCC, N),
]


@pytest.mark.parametrize("claim_table", [1, 2])
@pytest.mark.parametrize("name,shape,boundary,n", CASES, ids=[c[0] for c in CASES])
def test_open_launches_match_oracle(name, shape, boundary, n, claim_table):
    g, o = build_both(shape, lambda L: models.diffusion_only(L, n), 19, boundary=boundary, persistent=-1,
                      claim_table=claim_table)
    for k in (1, 6):
        g.run_events(k)
        o.run_events(k)
        assert_same(g, o, (name, k))


def test_open_launches_in_a_compartment():
    shape = (128, 120, 100)
    lab = models.cell_labels(*shape, radius=90.0)

    def recipe(L):
        L.set_compartments(lab, 3)
        L.species_compartment(L.add_species(1e-12, N), 2)
        L.species_compartment(L.add_species(0.7e-12, 3000), 1)

    g, o = build_both(shape, recipe, 7, persistent=-1)
    g.run_events(9)
    o.run_events(9)
    assert_same(g, o)


@pytest.mark.parametrize("shape,boundary", [((320, 304, 300), 7), ((315, 301, 299), 0)])
def test_large_lattices_take_them_and_agree_with_tables(shape, boundary):
    # above 28 million voxels: the automatic choice (whole bricks: the lean tile
    # kernel up to 2.6 million walkers) against the molecule-list kernel with
    # claims in hash tables
    out = []
    for table in (0, 2):
        L = psc.Lattice(*shape, voxel_radius=1e-8, boundary=boundary)
        L.set_options(claim_table=table, tiles=-1 if table else 0, time_kernels=1)
        L.add_species(1e-12, N + 12345)
        L.add_species(0.9e-12, 700)
        L.populate(2)
        L.run_events(75)
        L.set_options(time_kernels=-1)
        L.run_events(80)
        out.append((L.unwrapped(0), L.unwrapped(1), L.kernel_times()))
        L.close()
    for s in (0, 1):
        assert np.array_equal(out[0][s][0], out[1][s][0]) and np.array_equal(out[0][s][1], out[1][s][1])
    kt = out[0][2]
    assert kt["tile_events"] > 30 if boundary else kt["claim_launches"] > 30
