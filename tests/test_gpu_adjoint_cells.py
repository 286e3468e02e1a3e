"""The adjoint with beam particles on nodes of the xi grid: the beam's order, its deposit, its push and
their reverses find a particle in the same cell, whichever side of the node rounding puts it."""
import numpy as np
import pytest

import synth
from test_adjoint import adjoint_case, theta_of

pytestmark = pytest.mark.gpu


def _nodes_in_dispute(nxi, ximax):
    """Nodes k dxi whose cell by the quotient is not that by the product with the reciprocal."""
    dxi, k = ximax / nxi, np.arange(1, nxi)
    xi = k * dxi
    return xi[np.floor(xi / dxi) != np.floor(xi * (nxi / ximax))]


def _gradient(cfg, theta, steps):
    import torch
    from paper_1411_3246_gb300 import build, wake
    build.build()
    nm_b = synth.beam_normals(cfg)
    nm_b[4, cfg.n_drive:] = 0.0  # every witness particle at the bunch's centre
    with wake.Adjoint(cfg, steps, 4, torch.from_numpy(synth.plasma_normals(cfg)).cuda(), torch.from_numpy(nm_b).cuda()) as a:
        obs = np.array(a.forward(theta, [1.0] * 4))
        return obs, np.array(a.backward([1.0, -0.5]))


@pytest.mark.parametrize("nxi", [77, 91, 148])
def test_witness_on_a_node_pipelined_equals_sequential(nxi, monkeypatch):
    """The witness centred on a node that the two formulas put into different cells.  Tolerances: those of
    the pipelined adjoint against the sequential one with a random beam (test_gpu_adjoint)."""
    cfg = adjoint_case(nr=16, nxi=nxi, n_beam=1024)
    nodes = _nodes_in_dispute(nxi, cfg.ximax)
    nodes = nodes[(nodes >= 6.0) & (nodes <= 9.0)]  # behind the driver (at 4), inside the box
    theta = theta_of(cfg)
    cfg.xi_d = 4.0
    theta[1] = next(float(x - 4.0) for x in nodes[::-1] if 4.0 + (x - 4.0) == x)  # the centre is the node to the bit
    out = []
    for pipe in ("1", "0"):
        monkeypatch.setenv("WAKE_ADJOINT_PIPELINE", pipe)
        out.append(_gradient(cfg, theta, 3))
    (o1, g1), (o0, g0) = out
    np.testing.assert_allclose(o1, o0, rtol=1e-11)
    assert np.abs(g1 - g0).max() <= 1e-9 * np.abs(g0).max(), (g1, g0)
