"""Every form a march or a step can run in, checked where the sizes of the other tests choose another: the rules
that choose are asserted (wake_forms), so a change of a rule shows here instead of emptying a test.

Tolerances, of the same comparisons elsewhere: FP64 marches 1e-10 of peak |E_z| in the linear case and carried FP64
beams 1e-9 (test_gpu_parity, test_gpu_cluster); a slipping FP64 beam 1e-7 (test_gpu_cluster); the density of a
mixed step (test_gpu_corners) 2^-24 of a cell for each of nr cells, and 1.2e-5.  A slipping mixed beam: its fields
are within 1e-5 of peak |E_z| for the same density (test_gpu_parity) and the density within 2e-5, so a force (three
fields) is within 1e-4 of the peak; a momentum moves by that force's time, a position by the momentum's, and each
rounds to FP32 twice a step.  (A particle that missed one push would lie a slip, ds / 2 gamma^2, behind: a thousand
times xi's tolerance.)"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
COORDS = ("x", "y", "xi", "ux", "uy", "uz")


@pytest.fixture(scope="module")
def wk():
    import torch
    from paper_1411_3246_gb300 import build, wake
    build.build()
    assert torch.cuda.is_available()
    return wake


def _cuda(a):
    import torch
    return None if a is None else torch.from_numpy(a).cuda()


@pytest.mark.parametrize("nr,ppc,ctas", [(31, 2, 1), (64, 2, 2), (64, 4, 4), (128, 8, 4), (256, 8, 8)])
def test_fp64_march_by_rings(wk, nr, ppc, ctas):
    _fp64_march(wk, nr, ppc, ctas)


@pytest.mark.parametrize("nr,ppc", [(128, 4), (33, 4), (129, 8), (151, 7), (1024, 2)])
def test_fp64_march_by_one_cta(wk, nr, ppc, monkeypatch):
    """The form of handles with many simulations: the tile width forced, which takes no clusters."""
    monkeypatch.setenv("WAKE_TILE_NT", "512")
    _fp64_march(wk, nr, ppc, 1)


def _fp64_march(wk, nr, ppc, ctas):
    cfg = synth.config_linear(nr=nr, nxi=48)
    cfg.ppc = ppc
    ref = oracle.march(cfg, oracle.plasma_init(cfg, None), oracle.nb_analytic(cfg))
    with wk.Simulations([cfg], wk.WAKE_FP64) as s:
        wk.wake_load_plasma(s.h, 0, None)
        wk.wake_plasma_march(s.h)
        assert wk.wake_forms(s.h, 0)[0] == ctas
        f = {k: v.cpu().numpy() for k, v in s.fields(0).items()}
        assert s.status(0) == wk.WAKE_OK
    for k in ("psi", "ez", "er", "bth"):
        assert np.abs(f[k] - ref[k]).max() <= 1e-10 * np.abs(ref["ez"]).max(), k


def test_fp64_steps_by_one_cta(wk, monkeypatch):
    """Warm blowout, 5 steps, against the oracle (the steps of test_gpu_cluster without a cluster)."""
    monkeypatch.setenv("WAKE_TILE_NT", "512")
    cfg = synth.config_blowout(n_beam=5003, nr=65, nxi=96)
    got, lost, bm, _, forms = _steps(wk, cfg, wk.WAKE_FP64, 5)
    assert forms == (1, 0)
    for i, k in enumerate(COORDS):
        assert np.abs(got[i] - bm[k]).max() <= 1e-9 * max(1.0, np.abs(bm[k]).max()), k
    assert np.array_equal(lost, bm["lost"] != 0)


def _steps(wk, cfg, prec, steps):
    """(state, lost, the oracle's beam and its last march's peak |E_z|, forms) after pipelined steps."""
    nm_p, nm_b = synth.plasma_normals(cfg), synth.beam_normals(cfg)
    pl, bm = oracle.plasma_init(cfg, nm_p), oracle.beam_init(cfg, nm_b)
    ref = oracle.run(cfg, pl, bm, steps)
    with wk.Simulations([cfg], prec) as s:
        wk.wake_load_plasma(s.h, 0, _cuda(nm_p))
        wk.wake_load_beam(s.h, 0, _cuda(nm_b))
        wk.wake_step(s.h, steps)
        assert wk.wake_step_kernel_ms(s.h) > 0
        forms = wk.wake_forms(s.h, 0)[1:]
        xyz, lost = s.beam(0)
        assert s.status(0) == wk.WAKE_OK, wk.wake_last_error()
    return xyz.cpu().numpy(), lost.cpu().numpy() != 0, bm, np.abs(ref["ez"]).max(), forms


def _slow(nr, nxi, ppc, n_beam):
    """A very weak cold driver of gamma 40, some of whose particles cross a cell within 8 steps.  (With stronger
    fields or longer steps the result is ill-conditioned: the oracle's own beam moves by 1e-2 when its positions are
    rounded to FP32; here by 1e-7, the rounding itself.)"""
    cfg = synth.config_linear(nr=nr, nxi=nxi, n0=0.02)
    cfg.ximax, cfg.ppc = 12.0, ppc
    cfg = synth.two_bunch(cfg, 0.3, 4.0, n_beam)
    cfg.gamma_b, cfg.ds, cfg.eps_n = 40.0, 10.0, 1e-3
    return cfg


def _crossed(cfg, bm):
    """Particles that are in another xi cell than at the start."""
    xi0, dxi = oracle.beam_init(cfg, synth.beam_normals(cfg))["xi"], cfg.ximax / cfg.nxi
    return int((np.floor(bm["xi"] / dxi) > np.floor(xi0 / dxi)).sum())


def test_fp64_slipping_steps_by_one_cta(wk, monkeypatch):
    monkeypatch.setenv("WAKE_TILE_NT", "512")
    cfg = _slow(64, 64, 4, 20001)
    got, lost, bm, _, forms = _steps(wk, cfg, wk.WAKE_FP64, 8)
    assert forms == (1, 0) and _crossed(cfg, bm) > 1000
    for i, k in enumerate(COORDS):
        assert np.abs(got[i] - bm[k]).max() <= 1e-7 * np.abs(bm[k]).max(), k
    assert np.array_equal(lost, bm["lost"] != 0)


# (nr, nxi, ppc, n_beam, forced tile, form): one CTA with node grids, clusters of tiles, wide clusters, grids by cells
@pytest.mark.parametrize("nr,nxi,ppc,n_beam,tile,forms", [
    (64, 64, 4, 20001, None, (1, 0)),
    (128, 64, 8, 20001, None, (1, 0)),
    (128, 64, 12, 20001, None, (8, 0)),
    (512, 40, 4, 20001, None, (1, 0)),
    (800, 40, 6, 20001, None, (2, 0)),
    (1030, 40, 20, 20001, None, (4, 0)),
    (1030, 40, 32, 20001, None, (8, 0)),
    (64, 16, 4, 33001, None, (1, 1)),
    (140, 16, 8, 33001, "512", (1, 1)),
])
def test_mixed_slipping_steps(wk, nr, nxi, ppc, n_beam, tile, forms, monkeypatch):
    if tile:
        monkeypatch.setenv("WAKE_TILE_NT", tile)
    cfg = _slow(nr, nxi, ppc, n_beam)
    got, lost, bm, peak, ran = _steps(wk, cfg, wk.WAKE_MIXED, 8)
    assert ran == forms and _crossed(cfg, bm) > 1000
    span, eps = 8 * cfg.ds, 16 * 2.0 ** -24
    du = span * 1e-4 * peak
    tols = dict(x=span * du / cfg.gamma_b + eps * np.abs(bm["x"]).max(), y=span * du / cfg.gamma_b + eps * np.abs(bm["y"]).max(),
                ux=du + eps * np.abs(bm["ux"]).max(), uy=du + eps * np.abs(bm["uy"]).max(), uz=du + 1e-10,
                xi=2 * span * du / cfg.gamma_b ** 2 + 1e-10)
    for i, k in enumerate(COORDS):
        tol = tols[k]
        assert np.abs(got[i] - bm[k]).max() <= tol, (k, np.abs(got[i] - bm[k]).max(), tol)
    assert (lost != (bm["lost"] != 0)).sum() <= 2  # a particle at the wall to rounding


@pytest.mark.parametrize("nr,ppc", [(140, 8), (300, 8)])
def test_density_by_cells_of_four_and_eight_rings_per_thread(wk, nr, ppc, monkeypatch):
    """As test_gpu_corners, where few steps of these sizes run in clusters otherwise."""
    monkeypatch.setenv("WAKE_TILE_NT", "512")
    cfg = synth.config_blowout(n_beam=24601, nr=nr, nxi=12)
    cfg.ppc = ppc
    cfg.n_d, cfg.n_w, cfg.sigma_r = 0.1, 0.05, 1.5
    nm_p, nm_b = synth.plasma_normals(cfg), synth.beam_normals(cfg)
    pl, bm = oracle.plasma_init(cfg, nm_p), oracle.beam_init(cfg, nm_b)
    oracle.run(cfg, pl, bm, 1)
    ref = oracle.beam_deposit(cfg, bm)
    with wk.Simulations([cfg], wk.WAKE_MIXED) as s:
        wk.wake_load_plasma(s.h, 0, _cuda(nm_p))
        wk.wake_load_beam(s.h, 0, _cuda(nm_b))
        wk.wake_step(s.h, 2)
        assert wk.wake_forms(s.h, 0)[1:] == (1, 1)
        nb = s.nb(0).cpu().numpy()
        assert s.status(0) == wk.WAKE_OK, wk.wake_last_error()
    assert np.abs(nb - ref).max() <= (nr * 2.0 ** -24 + 1.2e-5) * np.abs(ref).max()


@pytest.mark.parametrize("nr,ppc,ctas", [(128, 16, 8), (800, 6, 2), (1030, 32, 8)])
def test_a_mixed_cluster_s_wait_runs_out(wk, nr, ppc, ctas, monkeypatch):
    """WAKE_SPIN_LIMIT=0, as in test_gpu_faults: the clusters (of tiles, of the wide form) give up together, the
    status says so, and a fresh handle runs."""
    cfg = synth.config_blowout(n_beam=1 << 14, nr=nr, nxi=64)
    cfg.ppc = ppc
    for limit, status in (("0", wk.WAKE_ETIMEOUT), (None, wk.WAKE_OK)):
        if limit is None:
            monkeypatch.delenv("WAKE_SPIN_LIMIT")
        else:
            monkeypatch.setenv("WAKE_SPIN_LIMIT", limit)
        with wk.Simulations([cfg], wk.WAKE_MIXED) as s:
            wk.wake_load_plasma(s.h, 0, _cuda(synth.plasma_normals(cfg)))
            wk.wake_load_beam(s.h, 0, _cuda(synth.beam_normals(cfg)))
            wk.wake_step(s.h, 6)
            assert wk.wake_forms(s.h, 0)[1] == ctas
            assert s.status(0) == status
            xyz, lost = s.beam(0)
        if limit is None:
            assert np.isfinite(xyz.cpu().numpy()[:, lost.cpu().numpy() == 0]).all()
