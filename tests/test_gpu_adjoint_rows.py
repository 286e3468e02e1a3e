"""The adjoint's one-warp tridiagonal solves at row counts that do not fill the lanes: few rows, a last lane with
one row or none, several rows per lane, against the host build, which eliminates row by row.  Tolerances: those
of test_gpu_adjoint_equals_host_build."""
import numpy as np
import pytest

import adjoint_host
import synth
from test_adjoint import adjoint_case, theta_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nr", [2, 31, 32, 33, 65, 100, 129, 225, 256])
def test_gpu_adjoint_equals_host_build_at(nr):
    import torch
    from paper_1411_3246_gb300 import build, wake
    build.build()
    cfg = adjoint_case(nr=nr, nxi=40, n_beam=1024)
    theta, prof = theta_of(cfg), np.linspace(0.7, 1.3, 4)
    nm_p, nm_b = synth.plasma_normals(cfg), synth.beam_normals(cfg)
    dobs = np.array([1.0, -0.5])
    o_h, g_h = adjoint_host.gradient(cfg, 3, theta, prof, nm_p, nm_b, dobs)
    with wake.Adjoint(cfg, 3, 4, torch.from_numpy(nm_p).cuda(), torch.from_numpy(nm_b).cuda()) as a:
        o, g = np.array(a.forward(theta, prof)), np.array(a.backward(dobs))
    np.testing.assert_allclose(o, o_h, rtol=1e-10)
    assert np.abs(g - g_h).max() <= 1e-8 * np.abs(g_h).max(), (g, g_h)
