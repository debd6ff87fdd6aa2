"""Lattices where device memory is short.

A failed allocation of one lattice is not taken for an error of the next.
"""
import pytest

import models
import paper_1605_03726_gb300 as psc

pytestmark = pytest.mark.gpu


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
