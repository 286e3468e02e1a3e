"""Marches and pipelined steps shared by a cluster of CTAs against the FP64 oracle, at the sizes
where the sharing can go wrong: rings that do not divide by the CTAs, a last CTA with few rings,
two nodes, grids at the edges of the scans' and the tridiagonal solve's lane counts.

The forms chosen: FP64 from 128 rings (4 CTAs) and 512 (8), mixed from 1024 (4) and 1536 (8), while few
simulations or steps run.  Tolerances are those of the single-CTA forms (test_gpu_parity):
FP64 1e-10 of peak |E_z| (linear), mixed 1e-5; carried beams 1e-9 and 1e-8 (FP64)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wk():
    import torch
    from paper_1411_3246_gb300 import build, wake
    build.build()
    assert torch.cuda.is_available()
    return wake


def _linear(nr, nxi, ppc, slab):
    cfg = synth.config_slab_linear(nr=nr, nxi=nxi) if slab else synth.config_linear(nr=nr, nxi=nxi)
    cfg.ppc = ppc
    return cfg


@pytest.mark.parametrize("nr,ppc,slab", [(2, 64, 0), (31, 5, 0), (33, 4, 0), (129, 4, 0), (151, 7, 0), (129, 7, 1),
                                         (1024, 8, 0)])
def test_fp64_linear_march(wk, nr, ppc, slab):
    cfgs = [_linear(nr, 40, ppc, slab), _linear(nr, 33, ppc, slab)]
    with wk.Simulations(cfgs, wk.WAKE_FP64) as s:
        for i in range(2):
            wk.wake_load_plasma(s.h, i, None)
        wk.wake_plasma_march(s.h)
        for i, cfg in enumerate(cfgs):
            ref = oracle.march(cfg, oracle.plasma_init(cfg, None), oracle.nb_analytic(cfg))
            scale = np.abs(ref["ez"]).max()
            f = s.fields(i)
            assert s.status(i) == wk.WAKE_OK
            for k in ("psi", "ez", "er", "bth"):
                assert np.abs(f[k].cpu().numpy() - ref[k]).max() <= 1e-10 * scale, (i, k)


@pytest.mark.parametrize("nr,ppc,slab", [(205, 5, 0), (1021, 2, 0), (301, 13, 0), (301, 6, 1), (64, 24, 0), (33, 241, 0)])
def test_mixed_linear_march(wk, nr, ppc, slab):
    cfg = _linear(nr, 48, ppc, slab)
    with wk.Simulations([cfg], wk.WAKE_MIXED) as s:
        wk.wake_load_plasma(s.h, 0, None)
        wk.wake_plasma_march(s.h)
        f = s.fields(0)
        assert s.status(0) == wk.WAKE_OK
    ref = oracle.march(cfg, oracle.plasma_init(cfg, None), oracle.nb_analytic(cfg))
    scale = np.abs(ref["ez"]).max()
    for k in ("psi", "ez", "er", "bth"):
        assert np.abs(f[k].cpu().numpy() - ref[k]).max() <= 1e-5 * scale, k


@pytest.mark.parametrize("slab,nr,nxi,n_beam,steps", [(0, 65, 96, 5003, 5), (1, 65, 96, 5003, 5), (0, 40, 64, 3, 2),
                                                      (0, 131, 70, 40001, 21)])
def test_fp64_steps(wk, slab, nr, nxi, n_beam, steps):
    import torch
    cfg = synth.config_slab_blowout(n_beam=n_beam, nr=nr, nxi=nxi) if slab else synth.config_blowout(n_beam=n_beam, nr=nr, nxi=nxi)
    nm_p, nm_b = synth.plasma_normals(cfg), synth.beam_normals(cfg)
    pl, bm = oracle.plasma_init(cfg, nm_p), oracle.beam_init(cfg, nm_b)
    ref = oracle.run(cfg, pl, bm, steps)
    with wk.Simulations([cfg], wk.WAKE_FP64) as s:
        wk.wake_load_plasma(s.h, 0, torch.from_numpy(nm_p).cuda())
        wk.wake_load_beam(s.h, 0, torch.from_numpy(nm_b).cuda())
        wk.wake_step(s.h, steps)
        xyz, lost = s.beam(0)
        f = s.fields(0)
        assert s.status(0) == wk.WAKE_OK, wk.wake_last_error()
    got = xyz.cpu().numpy()
    for i, k in enumerate(("x", "y", "xi", "ux", "uy", "uz")):
        assert np.abs(got[i] - bm[k]).max() <= 1e-9 * max(1.0, np.abs(bm[k]).max()), k
    assert np.array_equal(lost.cpu().numpy() != 0, bm["lost"] != 0)
    scale = np.abs(ref["ez"]).max()
    assert np.abs(f["ez"].cpu().numpy() - ref["ez"]).max() <= 1e-8 * scale


def test_fp64_steps_with_slipping_particles(wk):
    """Few steps of a slow beam (gamma 40: half of it crosses a cell within the launch), so that every
    CTA of a cluster makes and takes entries of the lists of slipped particles.  A relative change
    of 6e-8 in the beam's positions moves these results by up to 9e-3 (the oracle's own), so FP64
    rounding moves them by about 1e-10 at most; 1e-7 of each coordinate's largest value is allowed."""
    import torch
    cfg = synth.config_blowout(n_beam=20001, nr=64, nxi=64)
    cfg.gamma_b, cfg.n_d, cfg.n_w, cfg.ds = 40.0, 0.05, 0.0266, 40.0
    nm_p, nm_b = synth.plasma_normals(cfg), synth.beam_normals(cfg)
    pl, bm = oracle.plasma_init(cfg, nm_p), oracle.beam_init(cfg, nm_b)
    xi0 = bm["xi"].copy()
    oracle.run(cfg, pl, bm, 8)
    with wk.Simulations([cfg], wk.WAKE_FP64) as s:
        wk.wake_load_plasma(s.h, 0, torch.from_numpy(nm_p).cuda())
        wk.wake_load_beam(s.h, 0, torch.from_numpy(nm_b).cuda())
        wk.wake_step(s.h, 8)
        assert wk.wake_step_kernel_ms(s.h) > 0  # pipelined, not the separate calls
        xyz, lost = s.beam(0)
        assert s.status(0) == wk.WAKE_OK, wk.wake_last_error()
    dxi = cfg.ximax / cfg.nxi
    assert (np.floor(bm["xi"] / dxi) > np.floor(xi0 / dxi)).sum() > 1000  # cells are crossed
    got = xyz.cpu().numpy()
    for i, k in enumerate(("x", "y", "xi", "ux", "uy", "uz")):
        assert np.abs(got[i] - bm[k]).max() <= 1e-7 * np.abs(bm[k]).max(), k
    assert np.array_equal(lost.cpu().numpy() != 0, bm["lost"] != 0)
