"""Members of a batch that come and go between stretches.

The batch keeps the list lengths a stretch ended with for the next one.  They
belong to the member as it was then: a lattice that left the batch (and ran on
alone, or was destroyed, its address perhaps given to the next lattice) must
not be judged by them.  With births a stale pair of next id and event index
would put the member beyond the ids that stretches hold, and leave it in
launches per event phase for good.  A lattice that carries an error keeps it
when it joins a batch.
"""
import gc

import numpy as np
import pytest

import models
import paper_1605_03726_gb300 as psc

pytestmark = pytest.mark.gpu

TAU = 6.666666666666667e-05             # hop interval at D = 1 um^2/s, r_v = 10 nm
SHAPE = (24, 24, 24)


def splitting(stream, seed):
    """A splits into A + C, and takes C away again."""
    L = psc.Lattice(*SHAPE, voxel_radius=1e-8, stream=stream)
    L.set_options(claim_table=1, resort_period=-1)
    a = L.add_species(1e-12, 60)
    c = L.add_species(0.0, 0)
    L.add_reaction([a], [a, c], 0.002 / TAU)
    L.add_reaction([a, c], [a], 1e-19)
    L.populate(seed)
    return L


def events_in_stretches(B, n):
    before = B.launches()
    B.run_events(n)
    return B.launches() - before == 1                    # (per event phase: four or more an event)


def test_member_that_ran_alone_meanwhile_goes_on_in_stretches():
    import torch
    stream = torch.cuda.Stream().cuda_stream
    B = psc.Batch(stream=stream)
    L, solo = splitting(stream, 3), splitting(None, 3)
    B.add(L)
    assert events_in_stretches(B, 2)
    B.remove(L)
    # 8192 births an event at most: enough events for 2^27 ids
    L.run_events(17000)
    B.add(L)
    assert events_in_stretches(B, 2)                  # (takes up what the last stretch left)
    assert events_in_stretches(B, 100)
    solo.run_events(17104)
    assert np.array_equal(L.grid(), solo.grid()) and np.array_equal(L.counts(), solo.counts())
    B.close()


def test_new_members_do_not_inherit_list_lengths():
    import torch
    stream = torch.cuda.Stream().cuda_stream
    B = psc.Batch(stream=stream)
    for r in range(6):                                   # addresses come back
        L, solo = splitting(stream, r), splitting(None, r)
        B.add(L)
        assert events_in_stretches(B, 2), r
        assert events_in_stretches(B, 300), r
        solo.run_events(302)
        assert np.array_equal(L.counts(), solo.counts()), r
        B.remove(L)
        L.close()
        solo.close()
    B.close()


def test_many_short_calls():
    # list lengths come in the background, members join, leave and differ in their
    # options between calls; more members than one launch has blocks for
    import torch
    stream = torch.cuda.Stream().cuda_stream
    B = psc.Batch(stream=stream)
    members = [(splitting(stream, r), r) for r in range(170)]
    for L, r in members:
        B.add(L)
    late, _ = members[-1]
    B.remove(late)
    for call in range(150):
        if call == 40:
            B.add(late)
        if call == 90:
            members[0][0].set_options(collect_stats=1)
        B.run_events(1 + call % 2)
    for L, r in (members[0], members[85], members[-1]):
        solo = splitting(None, r)
        solo.run_events(L.event_index())
        assert L.event_index() == (225 if L is not late else 165)
        assert np.array_equal(L.grid(), solo.grid()) and np.array_equal(L.counts(), solo.counts())
        solo.close()
    attempts = members[0][0].stats()["attempts"]
    assert attempts > 100 * 30 and members[1][0].stats()["attempts"] == 0
    B.close()


def test_error_stays_with_a_lattice_that_joins_a_batch():
    import torch
    stream = torch.cuda.Stream().cuda_stream
    B = psc.Batch(stream=stream)
    L = psc.Lattice(48, 48, 48, voxel_radius=1e-8, stream=stream)
    L.set_options(claim_table=1, barrier_timeout_us=20000, barrier_phantom=1)
    L.add_species(1e-12, 3000)
    L.populate(17)
    L.run_events(4)                                      # a barrier that awaits a block that is not there
    with pytest.raises(psc.EngineError) as err:
        L.synchronize()
    assert err.value.rc == psc.E_TIMEOUT
    L.set_options(barrier_phantom=-1)
    g = L.event_index()
    gc.collect()                                         # no other lattice goes through these
    none = psc.ALLOC_FN(lambda nbytes, device, stream, ctx: None)
    no_free = psc.FREE_FN(lambda ptr, device, stream, ctx: None)
    assert psc.lib().psc_set_allocator(none, no_free, None) == psc.OK
    try:
        B.add(L)                                         # no room for the buffers of stretches
    finally:
        psc.use_cuda_malloc()
    B.run_events(3)
    assert L.event_index() == g
    with pytest.raises(psc.EngineError) as err:
        L.counts()
    assert err.value.rc == psc.E_TIMEOUT
    B.close()
    L.close()


def test_members_take_turns_where_their_cells_exceed_the_cache():
    # 136 MB of cells, 1.9 million molecules
    import torch
    stream = torch.cuda.Stream().cuda_stream

    def member(r, stream):
        L = psc.Lattice(100, 96 + 2 * (r % 3), 104, voxel_radius=1e-8, stream=stream)
        L.set_options(claim_table=1, resort_period=-1)
        if r % 2:
            models.reaction_diffusion_ab(L, 56000, 56000)
        else:
            models.diffusion_only(L, 56000, D=1e-12)
        L.populate(r)
        return L

    B = psc.Batch(stream=stream)
    members = [member(r, stream) for r in range(34)]
    for L in members:
        B.add(L)
    B.run_events(1)
    assert B.launches() > 1
    B.run_events(42)
    for r in (0, 1, 16, 17, 32, 33):
        solo = member(r, None)
        solo.run_events(43)
        assert np.array_equal(members[r].grid(), solo.grid())
        assert np.array_equal(members[r].unwrapped(0)[0], solo.unwrapped(0)[0])
        solo.close()
    B.close()


@pytest.mark.parametrize("members,n,births", [(153, 500, False), (310, 150, False), (310, 150, True)])
def test_more_members_than_blocks(members, n, births):
    # narrower blocks, two or four on an SM; options of a member changed on the way
    import torch
    stream = torch.cuda.Stream().cuda_stream

    def member(r, stream):
        L = psc.Lattice(20 + 2 * (r % 3), 20, 22, voxel_radius=1e-8, stream=stream)
        L.set_options(claim_table=1, resort_period=-1)
        a = L.add_species(1e-12, n)
        b = L.add_species(0.8e-12, n // 2)
        c = L.add_species(0.0, 5)
        L.add_reaction([a, b], [c, b], 1e-19)
        L.add_reaction([b], [a, b] if births else [a], 0.01 / TAU)
        L.populate(r)
        return L

    B = psc.Batch(stream=stream)
    Ls = [member(r, stream) for r in range(members)]
    for L in Ls:
        B.add(L)
    for k in (1, 3, 60, 1):
        B.run_events(k)
        Ls[7].set_options(collect_stats=1)
    for r in range(0, members, members // 9):
        solo = member(r, None)
        solo.run_events(65)
        assert np.array_equal(Ls[r].grid(), solo.grid()) and np.array_equal(Ls[r].counts(), solo.counts())
        for s in range(3):
            assert np.array_equal(Ls[r].unwrapped(s)[0], solo.unwrapped(s)[0])
        solo.close()
    assert Ls[7].stats()["attempts"] > 0
    B.close()
