"""The pipelined steps' density grids: calls that differ in length and in the grids' layout share one pool, which
only grows, and equal calls decide alike."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_calls_of_different_length_keep_the_pool():
    """A dense beam: 40 steps keep the grids by cells, 3 steps run in clusters with node grids."""
    import torch
    from paper_1411_3246_gb300 import build, wake
    build.build()
    cfg = synth.config_blowout(n_beam=2100 * 100, nr=200, nxi=100)
    cfg.ppc = 8
    nm = torch.from_numpy(synth.beam_normals(cfg)).cuda()
    with wake.Simulations([cfg], wake.WAKE_MIXED) as s:
        wake.wake_load_plasma(s.h, 0, torch.from_numpy(synth.plasma_normals(cfg)).cuda())
        free = []
        for steps in (40, 3, 40, 3, 40):
            wake.wake_load_beam(s.h, 0, nm)
            wake.wake_step(s.h, steps)
            assert s.status(0) == wake.WAKE_OK, wake.wake_last_error()
            free.append(torch.cuda.mem_get_info()[0])
    assert free[1:] == [free[1]] * 4, np.array(free) - free[1]
