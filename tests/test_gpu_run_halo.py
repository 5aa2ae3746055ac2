"""Grid.run leaves the halo cells of intermediate states out of date on the TMA
kernel (the stencil reads the neighbours' points instead): both buffers end bit
for bit as after steps that each update the halo."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

# tiles are 64 (FP64) or 128 points by 16 rows; the cases have one, two and
# several tiles per dimension, self-neighbours, rings, overlap 3, small grids
CASES = [((136, 36, 20), (2, 2, 2), (1, 0, 0), (2, 2, 2)),
         ((264, 40, 9), (1, 2, 2), (1, 1, 1), (2, 3, 2)),
         ((136, 18, 8), (3, 1, 1), (0, 0, 0), (3, 2, 2)),
         ((136, 19, 8), (1, 2, 1), (0, 1, 0), (2, 2, 2)),
         ((64, 24, 24), (2, 2, 2), (0, 0, 0), (2, 2, 2)),
         ((160, 50, 70), (2, 1, 2), (1, 1, 0), (3, 3, 3))]


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,dims,periods,overlap", CASES)
def test_run_equals_steps_with_halo_updates(n, dims, periods, overlap, dtype):
    import paper_2211_15716_gb300 as igg
    with igg.Grid(n, dims=dims, periods=periods, overlap=overlap) as g:
        ng = g.global_size()
        T0, Ci = np.empty(g.shape), np.empty(g.shape)
        for s in range(g.nsub):
            gi = g.global_indices(s)
            T0[s] = synth.sine_modes(2, *gi, ng, base=0.0)  # fix-ups next to the faces, too
            Ci[s] = synth.ci_uniform_c0(2, *gi, ng)
        T0[0] *= 1.01  # halo cells that disagree with their sources at the start
        T = torch.from_numpy(T0).to(dtype).cuda()
        C = torch.from_numpy(Ci).to(dtype).cuda()
        dd = (0.1, 0.08, 0.09)
        dt = min(d * d for d in dd) / 6.1 / float(C.float().max())
        for nt in (4, 5, 9, 40):
            A, B = T.clone(), T.clone()
            for _ in range(nt):
                g.step(B, A, C, 1.0, dt, *dd)
                g.update_halo(B)
                A, B = B, A
            X, Y = T.clone(), T.clone()
            assert g.run(nt, X, Y, C, 1.0, dt, *dd) is (X if nt % 2 == 0 else Y)
            if nt % 2:
                X, Y = Y, X
            assert g.device_status() == 0
            assert torch.equal(X, A), (nt, (X != A).sum().item())
            assert torch.equal(Y, B), (nt, (Y != B).sum().item())
