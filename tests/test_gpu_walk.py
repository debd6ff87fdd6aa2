"""Stretches of lattices without reactions (claim words that tell vacancy,
every molecule in shared memory), bit for bit against the oracle.

Sizes on either side of its shapes: one cluster up to 16,384 molecules, a block
per SM above, one molecule per thread of that grid and one more, eight per
thread (a batch of read-backs) and one more; extents of 3 and 4 across a
periodic wrap; ragged and mixed walls, FCC, several species among crowders;
other kernels in between, which want the claim words free; and the claims'
epochs used up within a run.
"""
import numpy as np
import pytest

import paper_1605_03726_gb300 as psc
from test_gpu_parity import assert_same, build_both

pytestmark = pytest.mark.gpu


def walkers(*species):
    return lambda L: [L.add_species(d, n) for d, n in species]


CASES = [
    ("cluster_edge", (40, 36, 44), 7, walkers((1e-12, 16384)), (1, 70)),
    ("grid_edge", (40, 36, 44), 7, walkers((1e-12, 16385)), (1, 70)),
    ("one_each", (128, 64, 64), 7, walkers((1e-12, 155648)), (3, 20)),
    ("one_more", (129, 63, 67), 0, walkers((1e-12, 155649)), (3, 20)),
    ("eight_more", (160, 128, 96), 7, walkers((1e-12, 8 * 155648 + 1)), (6,)),
    ("thin_wrap", (3, 4, 4), 7, walkers((1e-12, 17)), (300,)),
    ("full", (8, 6, 4), 7, walkers((1e-12, 8 * 6 * 4)), (5,)),
    ("one", (5, 7, 9), 0, walkers((1e-12, 1)), (200,)),
    ("ragged_mixed", (37, 30, 23), 2, walkers((0.0, 4000), (1e-12, 6000), (3e-12, 900)), (1, 130)),
    ("fcc", (41, 28, 36), 7 | psc.FCC, walkers((2e-12, 9000), (2e-12, 300)), (1, 130)),
    ("fcc_walls", (33, 27, 31), psc.PERIODIC_I | psc.FCC, walkers((1e-12, 14000)), (90,)),
    ("large_few", (320, 304, 290), 5, walkers((1e-12, 20000), (0.4e-12, 300)), (1, 130)),
    ("sorted_two", (96, 80, 64), 7, walkers((1e-12, 210000), (0.8e-12, 205000), (0.0, 30000)), (70, 90)),
]


@pytest.mark.parametrize("name,shape,boundary,recipe,calls", CASES, ids=[c[0] for c in CASES])
def test_walk_stretches_match_oracle(name, shape, boundary, recipe, calls):
    g, o = build_both(shape, recipe, 23, boundary=boundary)
    launches = g.stats()["launches"]
    for n in calls:
        g.run_events(n)
        o.run_events(n)
    assert g.stats()["launches"] - launches < 40                # stretches, not per-event launches
    assert_same(g, o, name)


def test_other_kernels_in_between():
    # per-event launches, the tile kernel, the molecule-list kernel and kernel
    # timing between stretches; the claim words change their meaning each time
    g, o = build_both((48, 44, 40), walkers((1e-12, 12000), (0.0, 3000)), 5)
    for opt in (dict(persistent=-1), dict(persistent=1), dict(tiles=1), dict(tiles=-1), dict(run_per_thread=8),
                dict(run_per_thread=-1), dict(time_kernels=1), dict(time_kernels=-1)):
        g.set_options(**opt)
        g.run_events(9)
        o.run_events(9)
        assert_same(g, o, opt)


def test_statistics_and_batches():
    stats = {}
    for persistent in (1, -1):
        L = psc.Lattice(48, 44, 40, voxel_radius=1e-8)
        L.set_options(collect_stats=1, persistent=persistent)
        L.add_species(1e-12, 20000)
        L.populate(5)
        L.run_events(40)
        stats[persistent] = {k: L.stats()[k] for k in ("attempts", "hops", "events")}
        L.close()
    assert stats[1] == stats[-1]
    # a member whose claim words told vacancy before it joined a batch
    import torch
    stream = torch.cuda.Stream()
    B = psc.Batch(stream=stream.cuda_stream)
    pair = []
    for st in (stream.cuda_stream, None):
        L = psc.Lattice(30, 32, 28, voxel_radius=1e-8, stream=st)
        L.set_options(claim_table=1, resort_period=-1)
        L.add_species(1e-12, 5000)
        L.populate(8)
        L.run_events(11)
        pair.append(L)
    B.add(pair[0])
    B.run_events(10)
    B.remove(pair[0])
    pair[0].run_events(5)
    pair[1].run_events(15)
    a, b = pair[0].coords(0), pair[1].coords(0)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    B.close()


def test_claims_epochs_run_out():
    # 2.1 million ids take 22 bits of a claim, which leaves 1022 epochs
    out = []
    for persistent in (1, -1):
        L = psc.Lattice(160, 160, 160, voxel_radius=1e-8)
        L.set_options(persistent=persistent)
        L.add_species(1e-12, (1 << 21) + 5)
        L.populate(3)
        for n in (1000, 700, 400):
            L.run_events(n)
        out.append(L.unwrapped(0))
        L.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


def test_stretches_of_some_of_the_species():
    # only the species with events in a stretch take part in it: calls of one event,
    # in a cluster or a grid by the species due, one without molecules among them
    recipe = walkers((1e-12, 40000), (0.9e-12, 300), (1.7e-12, 0), (0.0, 9000), (0.3e-12, 17000))
    g, o = build_both((64, 60, 62), recipe, 31, boundary=5)
    for n in (1,) * 12 + (3, 40, 1):
        g.run_events(n)
        o.run_events(n)
        assert_same(g, o, n)
