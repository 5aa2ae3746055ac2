"""The row-copy kernel (rows that are no multiple of 16 bytes): the bits of the
scalar kernel on row lengths around its tile widths and at every alignment of
the row starts, and an FP64 run against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

# 32 points is the shortest row it takes; FP64 tiles are 128 points by 8
# rows (the other types take the scalar kernel); one, two and three weight
# groups come from the spacings
CASES = [((33, 5, 4), (1, 1, 1)), ((35, 11, 9), (2, 1, 1)), ((127, 10, 6), (1, 2, 1)),
         ((129, 19, 7), (1, 1, 2)), ((131, 18, 5), (2, 2, 1)), ((259, 35, 20), (1, 1, 1)),
         ((31, 9, 6), (2, 1, 1))]
SPACINGS = [(0.1, 0.1, 0.1), (0.1, 0.08, 0.08), (0.1, 0.08, 0.09)]


def _fields(g, seed, dtype, base):
    ng = g.global_size()
    T0, Ci = np.empty(g.shape), np.empty(g.shape)
    for s in range(g.nsub):
        gi = g.global_indices(s)
        T0[s] = synth.sine_modes(seed, *gi, ng, base=base)
        Ci[s] = synth.ci_uniform_c0(seed, *gi, ng)
    return torch.from_numpy(T0).to(dtype).cuda(), torch.from_numpy(Ci).to(dtype).cuda()


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,dims", CASES)
def test_rows_kernel_gives_the_scalar_kernels_bits(n, dims, dtype):
    import paper_2211_15716_gb300 as igg
    for k, dd in enumerate(SPACINGS):
        out = []
        with igg.Grid(n, dims=dims, periods=(1, 0, 0)) as g:
            # base 0: stencils across zero and powers of two (FP64 fix-up)
            T, Ci = _fields(g, 5 + k, dtype, 0.0 if k else 1.7)
            dt = min(d * d for d in dd) / float(Ci.float().max()) / 6.1
            for tma in (1, 0):
                g.set_option(g.OPT_TMA, tma)
                out.append(g.run(5, T.clone(), T.clone(), Ci, 1.0, dt, *dd).clone())
                assert g.device_status() == 0
        assert torch.equal(out[0], out[1]), (dd, (out[0] != out[1]).sum().item())


def test_rows_kernel_fp64_matches_oracle():
    import paper_2211_15716_gb300 as igg
    n, dims = (67, 21, 19), (2, 1, 2)
    with igg.Grid(n, dims=dims) as g:
        T, Ci = _fields(g, 3, torch.float64, 1.7)
        dd = (0.1, 0.08, 0.09)
        dt = min(d * d for d in dd) / float(Ci.max()) / 6.1
        res = g.run(7, T.clone(), T.clone(), Ci, 1.0, dt, *dd).cpu().numpy()
    ref = oracle.run_decomposed(T.cpu().numpy(), Ci.cpu().numpy(), 7, 1.0, dt, *dd, dims, (0, 0, 0),
                                (2, 2, 2))
    assert np.abs(res - ref).max() <= 1e-12 * np.abs(ref).max()
