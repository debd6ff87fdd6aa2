"""Stretches of events of any species in one launch (short lists): one cluster
of blocks up to 16,384 molecules, a cooperative grid above.

Compared bit for bit with the oracle where such a stretch can go wrong: lists
on either side of the cluster's limit and crossing it, calls that end a stretch
after 1, 2, 511 and 513 events, per-event launches in between (they want the
occupancy bits and codes that stretches leave behind, and change the lists behind
the cells), lists of more entries than threads carry, reactions fast enough that tombstones fill
the lists' room several times within a stretch, births, immobile partners,
compartments, and walkers between species with reactions.
"""
import numpy as np
import pytest

import models
import paper_1605_03726_gb300 as psc
from test_gpu_parity import assert_same, build_both

pytestmark = pytest.mark.gpu

TAU = 6.666666666666667e-05             # hop interval at D = 1 um^2/s, r_v = 10 nm


def flipping(L, n):
    """A and B turn into each other, 8 % of them per event, and meet an immobile X."""
    a = L.add_species(1e-12, n)
    b = L.add_species(0.9e-12, n // 3)
    x = L.add_species(0.0, n // 4)
    L.add_reaction([a], [b], 0.08 / TAU)
    L.add_reaction([b], [a], 0.08 / TAU)
    L.add_reaction([a, x], [x, b], 1e-19)
    L.add_reaction([b, x], [a, x], 1e-19)


def splitting(L, n):
    """A splits and recombines; C takes A away; walkers in between."""
    a = L.add_species(1e-12, n)
    c = L.add_species(0.7e-12, n // 2)
    w = L.add_species(0.8e-12, n // 2)
    L.add_reaction([a], [a, c], 0.02 / TAU)
    L.add_reaction([a, c], [a], 5e-20)
    assert w == 2


def crowded(L, n):
    """More molecules than a grid's threads carry, walkers among them, between crowders."""
    L.add_species(0.0, n)
    a = L.add_species(1e-12, n)
    b = L.add_species(0.8e-12, n // 4)
    c = L.add_species(0.9e-12, 0)
    L.add_species(1e-12, 2 * n)
    L.add_reaction([a, b], [c], 3e-20)
    L.add_reaction([c], [a, b], 0.05 / TAU)


CASES = [
    ("ab_16383", (64, 64, 64), 7, lambda L: models.reaction_diffusion_ab(L, 16383, 9000), (1, 2, 511)),
    ("ab_16385", (64, 64, 64), 7, lambda L: models.reaction_diffusion_ab(L, 16385, 16384), (1, 513)),
    ("flip_cluster", (40, 36, 44), 7, lambda L: flipping(L, 5000), (513, 2)),
    ("flip_grid", (72, 64, 60), 0, lambda L: flipping(L, 20000), (511, 1)),
    ("split_cluster", (37, 41, 29), 0, lambda L: splitting(L, 700), (2, 150)),
    ("split_grid", (60, 58, 64), 7, lambda L: splitting(L, 18000), (40, 1)),
    ("crowded", (96, 92, 100), 0, lambda L: crowded(L, 170000), (2, 60)),
    ("walkers", (48, 44, 52), 6, lambda L: [L.add_species(d, n) for d, n in ((1e-12, 17000), (1e-12, 3), (0.6e-12, 900))],
     (1, 513)),
]


@pytest.mark.parametrize("name,shape,boundary,recipe,calls", CASES, ids=[c[0] for c in CASES])
def test_stretches_match_oracle(name, shape, boundary, recipe, calls):
    g, o = build_both(shape, recipe, 11, boundary=boundary)
    for n in calls:
        g.run_events(n)
        o.run_events(n)
        assert_same(g, o, (name, n))
    # per-event launches, then a stretch again
    for persistent in (-1, 1):
        g.set_options(persistent=persistent)
        g.run_events(7)
        o.run_events(7)
        assert_same(g, o, (name, persistent))
    g.set_options(resort_period=-1)
    before = g.stats()["launches"]
    g.run_events(64)
    assert g.stats()["launches"] - before <= 2            # one stretch, not per-event launches


def test_stretches_count_events_as_launches_do():
    stats = {}
    for persistent in (1, -1):
        L = psc.Lattice(40, 36, 44, voxel_radius=1e-8)
        L.set_options(collect_stats=1, persistent=persistent)
        flipping(L, 3000)
        L.populate(5)
        L.run_events(300)
        stats[persistent] = L.stats()
        L.close()
    for k in ("attempts", "hops", "collisions", "accepted", "reactions2", "fires", "reactions1", "births", "events"):
        assert stats[1][k] == stats[-1][k], k
    assert stats[1]["launches"] < stats[-1]["launches"] // 10


def test_stretch_in_a_cell_with_compartments():
    shape = (40, 36, 32)
    lab = models.cell_labels(*shape, radius=28.0)
    g, o = build_both(shape, lambda L: models.receptor_binding(L, lab, 1500, 500, n_x=300, n_outside=900, koff=2e3), 4,
                      boundary=0)
    for n in (3, 400):
        g.run_events(n)
        o.run_events(n)
        assert_same(g, o, n)


def test_members_in_stretches_and_in_launches_together():
    # batches: a member that keeps per-event launches (persistent = -1) beside members
    # that run in stretches, calls longer than a stretch, a member without
    # reactions, and a batch larger than one launch has blocks for
    import torch
    stream = torch.cuda.Stream()
    B = psc.Batch(stream=stream.cuda_stream)
    pairs = []
    for r in range(310):
        e = 8 + 2 * (r % 5) if r >= 6 else (24, 30, 40, 26, 28, 34)[r]
        both = []
        for st in (stream.cuda_stream, None):
            L = psc.Lattice(e, e, e, voxel_radius=1e-8, stream=st)
            L.set_options(claim_table=1, resort_period=-1, persistent=-1 if r == 1 else 1)
            if r == 2:
                L.add_species(1e-12, 3000)
            else:
                models.reaction_diffusion_ab(L, int(0.06 * e ** 3), int(0.04 * e ** 3))
            L.populate(40 + r)
            both.append(L)
        B.add(both[0])
        pairs.append(both)
    for n in (3, 530):
        B.run_events(n)
        for r, (m, solo) in enumerate(pairs):
            if r > 8 and r % 29:
                continue
            solo.run_events(n)
            assert np.array_equal(m.grid(), solo.grid()) and m.time() == solo.time()
            for s in range(m.n_species):
                a, b = m.coords(s), solo.coords(s)
                assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    B.close()


@pytest.mark.parametrize("D,stretches", [(1e-12, True), (1e-11, False)])
def test_long_runs_of_walkers_leave_stretches(D, stretches):
    # many walkers among rare reactions: one of their events for two of the reacting
    # species', or a hundred in a row (the tile and molecule-list kernels take those)
    def lattice(**options):
        L = psc.Lattice(96, 92, 100, voxel_radius=1e-8)
        L.set_options(resort_period=-1, **options)
        models.reaction_diffusion_ab(L, 500, 500, D=1e-12 if stretches else 5e-14)
        L.add_species(D, 270000)
        L.populate(8)
        return L

    a, b = lattice(), lattice(persistent=-1)
    for n in (3, 230):
        before = a.stats()["launches"]
        a.run_events(n)
        launches = a.stats()["launches"] - before
        b.run_events(n)
        assert np.array_equal(a.grid(), b.grid())
        for s in range(4):
            assert np.array_equal(a.unwrapped(s)[0], b.unwrapped(s)[0])
    assert (launches <= 3) == stretches


@pytest.mark.parametrize("calls", [(1, 1, 2, 513, 3, 70), (513, 1, 2)])
@pytest.mark.parametrize("shape,n,partners", [((64, 60, 64), 500, 40000), ((36, 40, 44), 6000, 9000)])
def test_short_calls_with_long_lists_to_close_up(shape, n, partners, calls):
    # calls of few events close the lists up in a grid, longer ones in a cluster
    def recipe(L):
        a = L.add_species(1e-12, n)
        x = L.add_species(0.0, partners)
        y = L.add_species(0.0, 0)
        L.add_reaction([a, x], [a, y], 2e-20)
        L.add_reaction([a, y], [x, a], 1e-20)

    g, o = build_both(shape, recipe, 23)
    for k in calls:
        g.run_events(k)
        o.run_events(k)
        assert_same(g, o, k)


@pytest.mark.parametrize("n,per_event", [(12000, 0.3), (30000, 0.2), (700, 0.9), (33, 0.5)])
def test_thousands_of_births_per_event(n, per_event):
    # ids follow the parents' order, whichever block appends a birth
    def recipe(L):
        a = L.add_species(1e-12, n)
        c = L.add_species(0.0, 10)
        L.add_reaction([a], [a, c], -np.log(1.0 - per_event) / TAU)

    g, o = build_both((64, 60, 64), recipe, 77)
    for k in (1, 3, 4):
        g.run_events(k)
        o.run_events(k)
        assert_same(g, o, k)


@pytest.mark.parametrize("shape,recipe", [
    ((320, 304, 300), lambda L: L.add_species(1e-12, 20000)),
    ((200, 192, 180), lambda L: models.reaction_diffusion_ab(L, 3000, 3000)),
    ((200, 192, 180), lambda L: [models.reaction_diffusion_ab(L, 3000, 3000), L.add_species(1e-12, 50000)]),
    ((96, 92, 88), lambda L: L.add_species(1e-12, 230000))])
def test_first_calls_of_few_events(shape, recipe):
    # large lattices put stretches off, long lists their first sort, until enough events
    # are ahead: the same lattice whatever the calls
    arms = []
    for calls in ((1,) * 14 + (3, 22, 1), (40,), None):
        L = psc.Lattice(*shape, voxel_radius=1e-8)
        recipe(L)
        L.populate(9)
        if calls:
            for n in calls:
                L.run_events(n)
        else:
            t = L.tau(0)
            while L.event_index() < 40:
                L.run(min(L.time() + 0.6 * t, 1.0))
            if L.event_index() > 40:
                L.close()
                continue
        arms.append([L.grid()] + [L.unwrapped(s)[0] for s in range(L.n_species)])
        L.close()
    for arm in arms[1:]:
        for a, b in zip(arms[0], arm):
            assert np.array_equal(a, b)
