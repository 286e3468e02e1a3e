"""The largest grids the shared-memory marches take: their solves' row arrays leave room for 1,200 radial cells in
FP64 (the slab runs nowhere else), also when a launch marches a smaller grid, with longer row arrays for its size,
beside the largest.  Tolerance: that of the FP64 march against the oracle in the linear case (test_gpu_parity),
1e-10 of peak |E_z|."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [None, "512"])  # a cluster's CTAs, one CTA
@pytest.mark.parametrize("sizes", [(1200, 1195, 1190), (1196,)])
def test_fp64_slab_at_the_limit_of_shared_memory(sizes, tile, monkeypatch):
    from paper_1411_3246_gb300 import build, wake
    build.build()
    if tile:
        monkeypatch.setenv("WAKE_TILE_NT", tile)
    cfgs = [synth.config_slab_linear(nr=nr, nxi=10) for nr in sizes]
    for c in cfgs:
        c.ppc = 2
    with wake.Simulations(cfgs, wake.WAKE_FP64) as s:
        for i in range(len(cfgs)):
            wake.wake_load_plasma(s.h, i, None)
        wake.wake_plasma_march(s.h)
        for i, cfg in enumerate(cfgs):
            ref = oracle.march(cfg, oracle.plasma_init(cfg, None), oracle.nb_analytic(cfg))
            f = s.fields(i)
            assert s.status(i) == wake.WAKE_OK
            for k in ("psi", "ez", "er", "bth"):
                assert np.abs(f[k].cpu().numpy() - ref[k]).max() <= 1e-10 * np.abs(ref["ez"]).max(), (i, k)
