"""Claim and commit launches that skip the claims of hops no other molecule can
contest, bit for bit against the oracle and against the other kernels.

They take lists of 262,144 molecules and more on lattices of more than 28 million
voxels, of which at most 30 % are occupied.  The test of the twelve neighbours
can go wrong on bricks that line up across a periodic wrap and bricks that do not,
walls, partial bricks, FCC layers, an odd number of layers, compartments; with
both kinds of claims, few and many neighbours.  Lists on smaller lattices of the
same shapes, and denser ones, take claims for every hop: compared with the oracle.
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


LARGE = [
    ("bricks", (320, 304, 292), 7, N),
    ("partial_bricks", (306, 302, 308), 7, N + 77),              # ni and nj not multiples of 4 across the wrap
    ("partial_mixed", (309, 302, 305), psc.PERIODIC_I, N),
    ("walls", (311, 307, 301), 0, 1700000),
    ("fcc_odd_layers", (304, 302, 309), 7 | psc.FCC, N),
    ("fcc_walls", (311, 307, 301), psc.FCC, 1100000),
]


@pytest.mark.parametrize("claim_table", [1, 2])
@pytest.mark.parametrize("name,shape,boundary,n", LARGE, ids=[c[0] for c in LARGE])
def test_large_lattices_match_the_molecule_list_kernel(name, shape, boundary, n, claim_table):
    out = []
    for options in (dict(persistent=-1, claim_table=claim_table), dict(claim_table=2, tiles=-1)):
        L = psc.Lattice(*shape, voxel_radius=1e-8, boundary=boundary)
        L.set_options(**options)
        models.diffusion_only(L, n)
        L.populate(19)
        for k in (1, 70):                                # (a re-sort in between)
            L.run_events(k)
        out.append(L.unwrapped(0))
        L.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1]), name


def test_large_lattice_with_compartments_and_crowders():
    shape = (312, 304, 300)
    lab = (np.arange(shape[0] * shape[1] * shape[2], dtype=np.int64) // (shape[0] * shape[1]) // 3 % 3).astype(np.uint8)
    out = []
    for options in (dict(persistent=-1), dict(claim_table=2, tiles=-1)):
        L = psc.Lattice(*shape, voxel_radius=1e-8)
        L.set_options(**options)
        L.set_compartments(lab, 3)
        L.add_species(1e-12, N + 5, compartment=2)
        L.add_species(0.0, 1000000, compartment=2)
        L.add_species(0.7e-12, N, compartment=0)
        L.populate(7)
        L.run_events(30)
        out.append([L.unwrapped(s)[0] for s in range(3)])
        L.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("occupied", [0.29, 0.31])       # either side of the densest they take
def test_dense_large_lattices_match_the_tile_kernel(occupied):
    shape = (312, 304, 300)
    out = []
    for options in (dict(persistent=-1), dict(tiles=1)):
        L = psc.Lattice(*shape, voxel_radius=1e-8)
        L.set_options(**options)
        models.diffusion_only(L, int(occupied * shape[0] * shape[1] * shape[2]))
        L.populate(3)
        L.run_events(5)
        out.append(L.unwrapped(0)[0])
        L.close()
    assert np.array_equal(*out)
