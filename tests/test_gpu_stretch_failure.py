"""Waits of stretches of reaction events that run out, without a GPU fault.

The barriers between the phases of such a stretch are bounded in a grid and in a
batch member's group of blocks.  Here they await a block that does not exist:
the error reaches the host, the lattice or member keeps it and gets no further
events, and the other members of the batch end where they end alone.
"""
import time

import numpy as np
import pytest

import models
import paper_1605_03726_gb300 as psc

pytestmark = pytest.mark.gpu


def lattice(edge, n, seed, stream=None, **options):
    L = psc.Lattice(edge, edge, edge, voxel_radius=1e-8, stream=stream)
    L.set_options(claim_table=1, resort_period=-1, **options)
    models.reaction_diffusion_ab(L, n, n)
    L.populate(seed)
    return L


@pytest.mark.parametrize("edge,n", [(48, 2000), (64, 20000)])
def test_wait_of_a_stretch_runs_out_and_is_reported(edge, n):
    L = lattice(edge, n, 3, barrier_timeout_us=20000, barrier_phantom=1)
    t0 = time.monotonic()
    L.run_events(8)
    for call in (L.synchronize, lambda: L.run_events(1), L.counts):
        with pytest.raises(psc.EngineError) as err:
            call()
        assert err.value.rc == psc.E_TIMEOUT
    assert time.monotonic() - t0 < 10.0 and L.event_index() == 8
    L.close()
    a, b = lattice(edge, n, 3), lattice(edge, n, 3, persistent=-1)     # the device goes on
    for M in (a, b):
        M.run_events(8)
    assert np.array_equal(a.grid(), b.grid())


@pytest.mark.parametrize("members", [3, 200])            # groups of many blocks; of one, in two launches
def test_member_whose_wait_runs_out_leaves_the_others_alone(members):
    import torch
    stream = torch.cuda.Stream().cuda_stream
    B = psc.Batch(stream=stream)
    bad = members // 2
    Ls = [lattice(40, 3000, r, stream, **(dict(barrier_timeout_us=20000, barrier_phantom=1) if r == bad else {}))
          for r in range(members)]
    for L in Ls:
        B.add(L)
    t0 = time.monotonic()
    B.run_events(5)
    Ls[0].synchronize()                                  # (list lengths come in the background)
    for n in (30, 20):
        B.run_events(n)
    with pytest.raises(psc.EngineError) as err:
        Ls[bad].synchronize()
    assert err.value.rc == psc.E_TIMEOUT and time.monotonic() - t0 < 10.0
    assert Ls[bad].event_index() == 5                    # the time-out is seen with the list lengths
    for r in range(0, members, max(1, members // 8)):
        if r == bad:
            continue
        solo = lattice(40, 3000, r)
        solo.run_events(55)
        assert np.array_equal(Ls[r].grid(), solo.grid()) and np.array_equal(Ls[r].counts(), solo.counts())
        solo.close()
    B.close()
