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


def test_beam_conversions_round_to_nearest_even():
    """A beam taken in FP64 and given back by the mixed form: x, y, u_x and u_y rounded to FP32, xi and
    u_z to the float-float pair, as IEEE conversions give them, on ties, neighbours of powers of
    two, subnormal and overflowing FP32 values and signed zeros; and the particles at the wall."""
    import torch
    from paper_1411_3246_gb300 import build, wake
    build.build()
    rng = np.random.default_rng(3)
    base = np.concatenate([rng.standard_normal(4000) * 10.0 ** rng.integers(-44, 38, 4000), [0.0, -0.0, 1.0, -1.0, 2.0 ** -126,
                           2.0 ** -149, 2.0 ** -150, 1.5 * 2.0 ** -149, 3.4028235e38, 3.4028236e38, 2.0 ** 100]])
    f = base.astype(np.float32).astype(np.float64)
    ties = (f + np.nextafter(base.astype(np.float32), np.float32(np.inf)).astype(np.float64)) / 2
    with np.errstate(over="ignore"):
        v = np.concatenate([base, ties, np.nextafter(ties, np.inf), np.nextafter(ties, -np.inf)])
        v = v[np.isfinite(v)]
        n = v.size
        cfg = synth.config_blowout(n_beam=n, nr=33, nxi=71)
        xyz = np.stack([v, np.roll(v, 1), np.roll(v, 2), np.roll(v, 3), np.roll(v, 5), np.roll(v, 7)])
        edge = np.array([np.nextafter(cfg.rmax, 0), cfg.rmax, np.nextafter(cfg.rmax, 9), cfg.rmax * (1 - 1e-6), cfg.rmax * (1 + 1e-6)])
        xyz[0, :5], xyz[1, :5], xyz[2, :5] = edge, 0.0, 1.0
        ref = xyz.astype(np.float32).astype(np.float64)
        for q in (2, 5):
            hi = xyz[q].astype(np.float32).astype(np.float64)
            ok = np.isfinite(hi)
            ref[q, ok] = hi[ok] + (xyz[q, ok] - hi[ok]).astype(np.float32).astype(np.float64)
        lost = ~((xyz[2] >= 0) & (xyz[2] < cfg.ximax) & (np.sqrt(xyz[0] ** 2 + xyz[1] ** 2) < cfg.rmax))
    with wake.Simulations([cfg], wake.WAKE_MIXED) as s:
        wake.wake_set_beam(s.h, 0, torch.from_numpy(xyz).cuda())
        got, gl = s.beam(0)
        got, gl = got.cpu().numpy(), gl.cpu().numpy()
    assert np.array_equal(gl != 0, lost)
    for q in range(6):
        ok = np.isfinite(ref[q])
        if q in (2, 5):
            ok &= np.abs(ref[q]) < 1e38
        assert np.array_equal(got[q][ok], ref[q][ok]) and np.array_equal(np.signbit(got[q][ok]), np.signbit(ref[q][ok])), q
