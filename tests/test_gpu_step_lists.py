"""Pipelined steps of slipping beams, through every step kernel that keeps lists of slipped particles: a
launch with more steps than the GPU holds CTAs, so that a CTA takes a second step after its first (its
control words are the next step's again), against the same steps taken one call at a time."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wk():
    import torch
    from paper_1411_3246_gb300 import build, wake
    build.build()
    assert torch.cuda.is_available()
    return wake


def _carry(wk, cfg, prec, steps, pipelined):
    import torch
    nm_p, nm_b = synth.plasma_normals(cfg), synth.beam_normals(cfg)
    with wk.Simulations([cfg], prec) as s:
        wk.wake_load_plasma(s.h, 0, None if nm_p is None else torch.from_numpy(nm_p).cuda())
        wk.wake_load_beam(s.h, 0, torch.from_numpy(nm_b).cuda())
        if pipelined:
            wk.wake_step(s.h, steps)
            assert wk.wake_step_kernel_ms(s.h) > 0
        else:
            for _ in range(steps):
                wk.wake_beam_deposit(s.h)
                wk.wake_plasma_march(s.h)
                wk.wake_beam_push(s.h)
        xyz, lost = s.beam(0)
        assert s.status(0) == wk.WAKE_OK, wk.wake_last_error()
        return xyz.cpu().numpy(), lost.cpu().numpy()


def _slow_beam(nr, nxi, n_beam):
    """A weak driver of gamma 40, which slips 1/40 cell a step."""
    cfg = synth.config_linear(nr=nr, nxi=nxi)
    cfg.ximax = 12.0
    cfg = synth.two_bunch(cfg, 0.3, 4.0, n_beam)
    cfg.gamma_b, cfg.ds, cfg.eps_n = 40.0, 5.0, 1e-3
    return cfg


def test_fp64_wide_steps_with_slipping_particles(wk, monkeypatch):
    """The FP64 wide form.  60 FP64 steps of such a beam agree to 1e-8 with separate ones
    (test_gpu_pipeline); these are five times as many: 1e-7."""
    import torch
    monkeypatch.setenv("WAKE_TILE_NT", "-1")
    cfg = _slow_beam(12, 192, 1500)
    steps = 2 * torch.cuda.get_device_properties(0).multi_processor_count + 20  # at most 2 CTAs of 512 threads per SM
    (a, la), (b, lb) = (_carry(wk, cfg, wk.WAKE_FP64, steps, p) for p in (True, False))
    assert np.array_equal(la, lb)
    nm = synth.beam_normals(cfg)
    xi0 = np.where(np.arange(cfg.n_beam) < cfg.n_drive, cfg.xi_d + cfg.sigma_zd * nm[4], cfg.xi_w + cfg.sigma_zw * nm[4])
    dxi = cfg.ximax / cfg.nxi
    assert (np.floor(a[2] / dxi) - np.floor(xi0 / dxi))[la == 0].max() >= 2
    for x, y in zip(a, b):
        assert np.abs(x - y)[la == 0].max() <= 1e-7 * max(np.abs(y[la == 0]).max(), 1.0)
