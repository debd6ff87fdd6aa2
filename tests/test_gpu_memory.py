"""Lattices where device memory is short.

What only makes events faster (claim words in place of hash tables, the cells
of stretches) is given up where there is no room for it, and the lattice runs in
the kernels that do without; results stay the same.  A failed allocation of one
lattice is not taken for an error of the next.
"""
import gc

import numpy as np
import pytest

import models
import paper_1605_03726_gb300 as psc

pytestmark = pytest.mark.gpu


class Capped:
    """Device memory from PyTorch's caching allocator, at most `cap` bytes."""

    def __init__(self):
        import torch
        self.torch = torch
        self.cap = 1 << 60
        self.live = {}
        self.sizes = []
        self.hooks = (psc.ALLOC_FN(self.alloc), psc.FREE_FN(self.free))

    def used(self):
        return sum(self.live.values())

    def alloc(self, nbytes, device, stream, ctx):
        if self.used() + nbytes > self.cap:
            return None
        p = self.torch.cuda.caching_allocator_alloc(int(nbytes), device, stream or 0)
        self.live[p] = int(nbytes)
        self.sizes.append(int(nbytes))
        return p

    def free(self, ptr, device, stream, ctx):
        del self.live[ptr]
        self.torch.cuda.caching_allocator_delete(ptr)


@pytest.fixture
def memory():
    gc.collect()                                         # lattices of other tests go back where they came from
    m = Capped()
    assert psc.lib().psc_set_allocator(m.hooks[0], m.hooks[1], None) == psc.OK
    yield m
    psc.use_cuda_malloc()
    assert not m.live


def state(L):
    return [L.grid(), L.counts()] + [x for s in range(L.n_species) for x in L.coords(s) + L.unwrapped(s)]


def same(a, b):
    assert len(a) == len(b) and all(np.array_equal(x, y) for x, y in zip(a, b))


# one cluster; a grid, with scratch to close the lists up; room for the cells, not for that
@pytest.mark.parametrize("n,cells", [(2000, 0), (20000, 0), (20000, 1)])
def test_reactions_run_without_room_for_stretches(memory, n, cells):
    shape = (168, 168, 160)

    def lattice():
        L = psc.Lattice(*shape, voxel_radius=1e-8)
        models.reaction_diffusion_ab(L, n, n)
        L.populate(5)
        return L

    L = lattice()
    placed = memory.used()
    L.run_events(100)
    assert memory.used() > placed                        # the buffers of stretches
    expected = [state(L)]
    L.run_events(100)
    expected.append(state(L))
    L.close()
    memory.cap = placed + 65536 + cells * 4 * shape[0] * shape[1] * shape[2]
    L = lattice()
    before = L.stats()["launches"]
    L.run_events(100)
    memory.cap = 1 << 60                                 # (a grid's read-out takes a buffer for a while)
    same(state(L), expected[0])
    assert L.stats()["launches"] - before > 200          # a launch per phase
    L.set_options(resort_period=-1)                      # options ask again
    before = L.stats()["launches"]
    L.run_events(100)
    assert L.stats()["launches"] - before < 10
    same(state(L), expected[1])
    L.close()


@pytest.mark.parametrize("shape,n", [((200, 200, 192), 100000), ((400, 300, 240), 270000)])
def test_walkers_take_tables_without_room_for_claim_words(memory, shape, n):
    def lattice(**options):
        L = psc.Lattice(*shape, voxel_radius=1e-8)
        L.set_options(**options)
        models.diffusion_only(L, n)
        L.populate(5)
        return L

    L = lattice(claim_table=2)
    tables = memory.used()
    L.close()
    L = lattice()
    words = memory.used()
    L.run_events(40)
    expected = state(L)
    L.close()
    assert words > tables + (8 << 20)
    for cap in (words - 1, tables + (4 << 20)):          # a byte too little; room for tables only
        memory.cap = cap
        L = lattice()
        assert L.device_bytes() < tables + (4 << 20)
        memory.cap = 1 << 60                             # (the tile kernel's buffers)
        L.run_events(40)
        same(state(L), expected)
        L.close()


def test_failed_allocation_is_not_the_next_lattice_s_error():
    big = psc.Lattice(1290, 1290, 1290, voxel_radius=1e-8)
    a = big.add_species(1e-12, 100)
    for _ in range(8):                                   # lists of products sized for the lattice: 300 GB
        c = big.add_species(1e-12, 0)
        big.add_reaction([a], [a, c], 1.0)
    with pytest.raises(psc.EngineError) as err:
        big.populate(1)
    assert err.value.rc == psc.E_NOMEM
    L = psc.Lattice(48, 48, 48, voxel_radius=1e-8)
    models.reaction_diffusion_ab(L, 500, 500)
    L.populate(1)
    L.run_events(20)
    assert L.counts().sum() <= 1000 and len(L.coords(0)[1]) == L.counts()[0]
    L.close()
    big.close()
