"""Checkpointed runs on 3-D grids with an odd number of points: every other
state inside the drivers' FP64 buffers starts 8 bytes off a 16-byte boundary,
where the row-copy kernel's bulk copies cannot start."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

from paper_2211_15716_gb300 import autograd as ag  # noqa: E402


def _case(n):
    g = [np.arange(k) for k in n]
    Ci = np.ascontiguousarray(synth.ci_smooth(4, *g, n))
    T0 = np.ascontiguousarray(np.broadcast_to(synth.gaussian_bump(*g, n, sigma=0.15), Ci.shape))
    dd = [oracle.spacing(1.0, k) for k in n]
    return T0, Ci, dd, oracle.cfl_dt(*dd, 1.0, Ci.max())


def _dev(a):
    return torch.from_numpy(a.copy()).cuda().reshape(1, *a.shape)


# (33 points: the shortest rows of the row-copy kernel; 129: two tiles)
@pytest.mark.parametrize("n", [(65, 35, 33), (33, 5, 7), (129, 9, 11)])
@pytest.mark.parametrize("nt,every", [(7, 3), (6, 2), (5, 1)])
def test_gradient_matches_oracle(n, nt, every):
    import paper_2211_15716_gb300 as igg
    T0, Ci, dd, dt = _case(n)
    obs = 0.9 * T0
    _, gT0, gCi = oracle.gradient(T0, Ci, obs, nt, 1.0, dt, *dd)
    with igg.Grid(n) as g:
        T, C = _dev(T0).requires_grad_(True), _dev(Ci).requires_grad_(True)
        Tn = ag.solve(T, C, g, nt, 1.0, dt, *dd, every=every)
        gT, gC = torch.autograd.grad(Tn, (T, C), grad_outputs=ag.residual(Tn.detach(), _dev(obs)))
        gT, gC = gT.cpu().numpy()[0], gC.cpu().numpy()[0]
        assert g.device_status() == 0
    assert np.linalg.norm(gT - gT0) <= 1e-10 * np.linalg.norm(gT0)
    assert np.linalg.norm(gC - gCi) <= 1e-10 * np.linalg.norm(gCi)


def test_forward_gives_the_time_loops_bits_also_captured():
    import paper_2211_15716_gb300 as igg
    n, nt, every = (65, 35, 33), 7, 3
    T0, Ci, dd, dt = _case(n)
    with igg.Grid(n) as g:
        T, C = _dev(T0), _dev(Ci)
        ref = g.run(nt, T.clone(), T.clone(), C, 1.0, dt, *dd)  # (builds the tile tables)
        out, _ = ag.forward_checkpointed(g, nt, every, T, C, 1.0, dt, *dd)
        assert torch.equal(out, ref)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            out, _ = ag.forward_checkpointed(g, nt, every, T, C, 1.0, dt, *dd)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
        assert g.device_status() == 0
