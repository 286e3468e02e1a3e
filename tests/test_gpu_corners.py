"""The pipelined steps' density grids: the density the last march used against the oracle's deposit,
after one step (the launch's own deposit) and two (the shares pushed into the next grid).  Beams of
2,048 particles per xi cell and more keep them by cells, four corner shares each (mixed form).

Tolerance: a particle's radial offset is known to nr 2^-24 of a cell in FP32 (8e-6 at 140 cells) and
its shares to a few 2^-24; a node's sum of up to ~5,000 shares adds sqrt(5000) 2^-24 = 4e-6: 2e-5 of the
largest node."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_beam,nr,nxi,slab,steps", [(5003, 65, 40, 0, 2), (5003, 33, 64, 1, 2), (24601, 2, 12, 0, 1),
                                                      (24601, 65, 12, 0, 1), (24601, 65, 12, 0, 2), (24601, 140, 12, 0, 2)])
def test_density_of_the_last_march(n_beam, nr, nxi, slab, steps):
    import torch
    from paper_1411_3246_gb300 import build, wake
    build.build()
    cfg = synth.config_slab_blowout(n_beam=n_beam, nr=nr, nxi=nxi) if slab else synth.config_blowout(n_beam=n_beam, nr=nr, nxi=nxi)
    cfg.n_d, cfg.n_w, cfg.sigma_r = 0.1, 0.05, 1.5  # a weak wide beam: nodes from the axis to the wall
    nm_p, nm_b = synth.plasma_normals(cfg), synth.beam_normals(cfg)
    pl, bm = oracle.plasma_init(cfg, nm_p), oracle.beam_init(cfg, nm_b)
    if steps > 1:
        oracle.run(cfg, pl, bm, steps - 1)
    ref = oracle.beam_deposit(cfg, bm)
    with wake.Simulations([cfg], wake.WAKE_MIXED) as s:
        wake.wake_load_plasma(s.h, 0, torch.from_numpy(nm_p).cuda())
        wake.wake_load_beam(s.h, 0, torch.from_numpy(nm_b).cuda())
        wake.wake_step(s.h, steps)
        nb = s.nb(0).cpu().numpy()
        assert s.status(0) == wake.WAKE_OK, wake.wake_last_error()
    assert np.abs(nb - ref).max() <= 2e-5 * np.abs(ref).max()
