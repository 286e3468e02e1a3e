"""wake_beam_push_steps(n) takes a particle's n steps in one launch (64 at most per launch): the same
state, bit for bit, as n calls of wake_beam_push, whether the fields are gathered from the grids or
from packed nodes, with particles lost on the way."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form,slab,n_beam", [("mixed", 0, 5001), ("mixed", 0, 301), ("mixed", 1, 5001), ("fp64", 0, 1000),
                                              ("mixed64", 0, 5001)])
def test_fused_pushes_equal_single_ones(form, slab, n_beam):
    import torch
    from paper_1411_3246_gb300 import build, wake
    build.build()
    prec = dict(mixed=wake.WAKE_MIXED, fp64=wake.WAKE_FP64, mixed64=wake.WAKE_MIXED64)[form]
    cfg = synth.config_blowout(n_beam=n_beam, nr=33, nxi=71)  # 2,448 nodes
    cfg.geometry, cfg.gamma_b, cfg.sigma_r = slab, 30.0, 1.2
    nm_p = torch.from_numpy(synth.plasma_normals(cfg)).cuda()
    nm_b = torch.from_numpy(synth.beam_normals(cfg)).cuda()
    out = []
    for fused in (False, True):
        with wake.Simulations([cfg], prec) as s:
            dt = torch.float64 if form == "fp64" else torch.float32
            f = [torch.empty(cfg.nxi + 1, cfg.nr + 1, dtype=dt, device="cuda") for _ in range(4)]
            wake.wake_bind_fields(s.h, 0, *f)
            wake.wake_load_plasma(s.h, 0, nm_p)
            wake.wake_load_beam(s.h, 0, nm_b)
            wake.wake_beam_deposit(s.h)
            wake.wake_plasma_march(s.h)
            xi = torch.linspace(0, 1, cfg.nxi + 1, device="cuda")[:, None]
            r = torch.linspace(0, 1, cfg.nr + 1, device="cuda")[None, :]
            for t, v in zip(f[1:], (0.3 * torch.sin(9 * xi) * (1 - r), -0.4 * r * torch.cos(5 * xi), 0.2 * r + 0 * xi)):
                t.copy_(v)
            if fused:
                wake.wake_beam_push_steps(s.h, 67)
            else:
                for _ in range(67):
                    wake.wake_beam_push(s.h)
            xyz, lost = s.beam(0)
            out.append((xyz.cpu().numpy(), lost.cpu().numpy()))
    assert 0.02 * n_beam < out[0][1].sum() < n_beam  # some are lost, not all
    assert np.array_equal(out[0][1], out[1][1])
    assert np.array_equal(out[0][0], out[1][0])
