"""Grid.run on small grids (graphs of up to 16 steps, the last used ones kept) is
the same, bit for bit, as its steps one by one: runs of any number of steps one
after the other on the same buffers, and more buffers than graphs are kept."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("n,dims", [((24, 20, 16), (1, 1, 1)), ((24, 20, 16), (2, 1, 2)),
                                    ((200, 40, 12), (2, 2, 1))])  # (FP32: halo cells left stale)
def test_any_number_of_steps(n, dims, dtype):
    import paper_2211_15716_gb300 as igg
    rng = np.random.default_rng(5)
    dd = (0.1, 0.08, 0.09)
    with igg.Grid(n, dims=dims, periods=(1, 0, 0)) as g:
        C = torch.from_numpy(rng.uniform(0.4, 0.667, g.shape)).to(dtype).cuda()
        T = torch.from_numpy(1.7 + 0.2 * rng.uniform(-1, 1, g.shape)).to(dtype).cuda()
        g.update_halo(T)
        dt = min(d * d for d in dd) / 0.667 / 6.1
        A, B = T.clone(), T.clone()
        a, b = T.clone(), T.clone()
        for nt in (1, 2, 7, 16, 30, 33, 4, 50, 5):
            res = g.run(nt, A, B, C, 1.0, dt, *dd)
            if res is B:
                A, B = B, A
            for _ in range(nt):
                g.step(b, a, C, 1.0, dt, *dd)
                g.update_halo(b)
                a, b = b, a
            assert torch.equal(A, a), nt
            assert torch.equal(B, b), nt
        assert g.device_status() == 0


def test_more_graphs_than_are_kept():
    import paper_2211_15716_gb300 as igg
    rng = np.random.default_rng(6)
    dd = (0.1, 0.1, 0.1)
    with igg.Grid((16, 12, 10)) as g:
        C = torch.from_numpy(rng.uniform(0.4, 0.667, g.shape)).cuda()
        T0 = torch.from_numpy(1.7 + 0.2 * rng.uniform(-1, 1, g.shape)).cuda()
        dt = 0.1 * 0.1 / 0.667 / 6.1
        states = [T0]
        for _ in range(18):
            b = states[-1].clone()
            g.step(b, states[-1], C, 1.0, dt, *dd)
            states.append(b)
        bufs = [(T0.clone(), T0.clone()) for _ in range(40)]
        for nt in (2, 16, 2, 2):  # (80 graphs)
            for A, B in bufs:
                A.copy_(T0)
                B.copy_(T0)
                assert torch.equal(g.run(nt, A, B, C, 1.0, dt, *dd), states[nt])
        assert g.device_status() == 0
