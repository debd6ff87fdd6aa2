"""The lean tile kernel's queues: contested molecules are decided 32 at a time
per warp, departures go through an outbox of 512 per event.  Boxes with fewer
molecules than a warp, with a chunk of 1024 on either side, and dense ones whose
departures overflow the outbox, bit for bit with the oracle."""
import pytest

import models
import paper_1605_03726_gb300 as psc
from test_gpu_parity import assert_same, build_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,regions", [(1, 12), (300, 27), (12 * 1024, 12), (12 * 1030, 12), (200000, 8), (500000, 8)])
def test_lean_queues_match_oracle(n, regions):
    g, o = build_both((96, 96, 88), lambda L: models.diffusion_only(L, n), 7, boundary=psc.PERIODIC_I,
                      claim_table=1, tiles=1, tile_regions=regions, tile_lean=1, time_kernels=1)
    for chunk in (1, 20):
        g.run_events(chunk)
        o.run_events(chunk)
        assert_same(g, o, chunk)
    assert g.kernel_times()["tile_lean_events"] == 21
