"""The emulated FP64 cell at group sums from 2^45 to past 2^47 ulps (the fast
path takes them up to 2^47): every kernel gives the same bits, each point lies
within the paths' error bound of the exact rational update."""
from fractions import Fraction as Fr

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [66, 67, 200])
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("rel", [0.003, 0.012])
@pytest.mark.parametrize("dd", [(0.1, 0.1, 0.1), (0.1, 0.08, 0.08), (0.1, 0.08, 0.09)])
def test_wide_group_sums(dd, rel, sign, nx):
    import paper_2211_15716_gb300 as igg
    n = (nx, 21, 12)
    rng = np.random.default_rng(11)
    T0 = sign * 3.0 * (1 + rel * rng.uniform(-2, 2, (1, n[2], n[1], n[0])))  # in (2, 4)
    Ci = rng.uniform(0.4, 0.667, T0.shape)
    dt = min(d * d for d in dd) / 0.667 / 6.1
    outs = []
    with igg.Grid(n) as g:
        for tma in (1, 0):
            g.set_option(g.OPT_TMA, tma)
            T = torch.from_numpy(T0).cuda().view(g.shape)
            C = torch.from_numpy(Ci).cuda().view(g.shape)
            outs.append(g.run(1, T, T.clone(), C, 1.0, dt, *dd).cpu().numpy()[0])
        assert g.device_status() == 0
    assert np.array_equal(outs[0].view(np.int64), outs[1].view(np.int64))
    w = [Fr(dt * 1.0 / (d * d)) for d in dd]
    u = Fr(2) ** (1024 - 1075)
    # two roundings to T's ulp, half an ulp of the weights' roundings, and 2^-44
    # of Ci sum |w G| (the FP32 sums of the float pairs)
    for _ in range(400):
        z, y, x = (int(rng.integers(1, k - 1)) for k in (n[2], n[1], n[0]))
        t = [Fr(float(v)) for v in (T0[0, z, y, x], T0[0, z, y, x - 1], T0[0, z, y, x + 1],
                                    T0[0, z, y - 1, x], T0[0, z, y + 1, x], T0[0, z - 1, y, x],
                                    T0[0, z + 1, y, x])]
        d2 = [t[1 + 2 * d] + t[2 + 2 * d] - 2 * t[0] for d in range(3)]
        ci = Fr(float(Ci[0, z, y, x]))
        exact = t[0] + ci * sum(a * b for a, b in zip(w, d2))
        bound = Fr(5, 2) * u + Fr(2) ** -44 * ci * sum(a * abs(b) for a, b in zip(w, d2))
        assert abs(Fr(float(outs[0][z, y, x])) - exact) <= bound, (x, y, z)
