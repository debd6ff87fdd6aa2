"""The launches per event phase, and their replay from CUDA graphs, on small
lattices.

Lattices of up to 2^26 voxels run their reaction events in stretches, so these
kernels meet small lattices with a claim word per voxel only where stretches are
off (persistent = -1).  They still run longer lists and larger lattices.  Every
replay of a graph of several events writes the event index first, a launch
more than the launches it replays: the counts tell that graphs were replayed.
"""
import pytest

import models
import paper_1605_03726_gb300 as psc
from test_gpu_fuzz import random_model
from test_gpu_graphs import same, state
from test_gpu_parity import assert_same, build_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graphs", [-1, 16])
@pytest.mark.parametrize("seed", range(0, 64, 5))
def test_random_models_in_launches_per_phase(seed, graphs):
    shape, walls, recipe, n_rx = random_model(seed)
    g, o = build_both(shape, recipe, 100 + seed, boundary=walls, claim_table=1, persistent=-1, graph_events=graphs)
    before = g.stats()["launches"]
    for n in (60, 120):
        g.run_events(n)
        o.run_events(n)
        assert_same(g, o, (seed, n_rx, n))
    assert g.stats()["launches"] - before >= 180


def ab(L):
    models.reaction_diffusion_ab(L, 2000, 2000, k=1e-20)


def cell_hcp(L):
    models.receptor_binding(L, models.cell_labels(40, 36, 32, radius=28.0), 1200, 500, n_x=300, n_outside=1000, koff=2e3)


def cell_fcc(L):
    models.receptor_binding(L, models.cell_labels(37, 29, 23, radius=24.0), 1200, 500, n_x=300, n_outside=1000, koff=2e3)


@pytest.mark.parametrize("name,shape,boundary,recipe,ns,k",
                         [("ab", (64, 64, 64), 7, ab, 3, 16), ("ab", (64, 64, 64), 7, ab, 3, 32),
                          ("cell", (40, 36, 32), 0, cell_hcp, 5, 16), ("cell_fcc", (37, 29, 23), psc.FCC, cell_fcc, 5, 16)])
def test_graphs_of_direct_claims_are_replayed(name, shape, boundary, recipe, ns, k):
    # one more launch per replay than without graphs; new launch options drop
    # the graphs, and the pattern's new ones give the same lattice
    arms = []
    for graphs in (-1, k):
        g, o = build_both(shape, recipe, 6, boundary=boundary, claim_table=1, persistent=-1, resort_period=k,
                          graph_events=graphs)
        counts = []
        for threads in (256, 128):
            g.set_options(block_threads=threads)
            before = g.stats()["launches"]
            g.run_events(24 * k)
            o.run_events(24 * k)
            counts.append(g.stats()["launches"] - before)
            assert_same(g, o, (name, graphs, threads))
        arms.append((state(g, ns), counts))
        g.close()
    same(arms[0][0], arms[1][0], name)
    if name == "ab":                                     # (its lists keep their launch shapes)
        for plain, replayed in zip(arms[0][1], arms[1][1]):
            assert plain >= 24 * k * 3                   # claim, commit, list passes
            assert replayed > plain + 6
