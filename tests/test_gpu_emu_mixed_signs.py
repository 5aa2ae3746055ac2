"""FP64 steps of fields whose neighbouring points have unrelated signs and
sizes: their group sums reach 3 * 2^55 ulps of the stencil's largest value,
far past the 2^47 that the emulated cell's paths take, so nearly every point
must reach the FP64 cell, in every kernel."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# (70, 21, 19): one launch with the fix-up inside; (130, 130, 70): stencil and
# fix-up launches; (67, 21, 19): row-copy kernel; (31, 21, 19): scalar kernel
GRIDS = [(70, 21, 19), (130, 130, 70), (67, 21, 19), (31, 21, 19)]
# one, two and three weight groups
SPACINGS = [(0.1, 0.1, 0.1), (0.1, 0.08, 0.08), (0.1, 0.08, 0.09)]


def _step(T, Ci, w):
    c = T[1:-1, 1:-1, 1:-1]
    lap = (w[0] * (T[1:-1, 1:-1, :-2] + T[1:-1, 1:-1, 2:] - 2 * c)
           + w[1] * (T[1:-1, :-2, 1:-1] + T[1:-1, 2:, 1:-1] - 2 * c)
           + w[2] * (T[:-2, 1:-1, 1:-1] + T[2:, 1:-1, 1:-1] - 2 * c))
    out = T.copy()
    out[1:-1, 1:-1, 1:-1] += Ci[1:-1, 1:-1, 1:-1] * lap
    return out


def _field(kind, n, rng):
    s = (n[2], n[1], n[0])
    if kind == "uniform":
        return rng.uniform(-1, 1, s)
    if kind == "positive":  # one sign, many exponents
        return rng.uniform(0, 1, s)
    if kind == "signs":  # one size: group sums at multiples of 2^54 ulps
        return rng.choice([-1.0, 1.0], s) * rng.uniform(0.999, 1.0, s)
    # centres 1 among -1/3: equal spacings make the group sum -2^55 ulps
    z, y, x = np.indices(s)
    return np.where((x + y + z) % 2, -1.0 / 3.0, 1.0)


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("kind", ["uniform", "positive", "signs", "thirds"])
@pytest.mark.parametrize("dd", SPACINGS)
def test_step_matches_fp64(dd, kind, n):
    import paper_2211_15716_gb300 as igg
    rng = np.random.default_rng(17)
    T0 = _field(kind, n, rng)
    Ci = rng.uniform(0.4, 0.667, T0.shape)
    dt = min(d * d for d in dd) / 0.667 / 6.1
    ref = _step(T0, Ci, [dt / (d * d) for d in dd])
    with igg.Grid(n) as g:
        T = torch.from_numpy(T0).cuda().view(g.shape)
        C = torch.from_numpy(Ci).cuda().view(g.shape)
        outs = []
        for tma in (1, 0):
            g.set_option(g.OPT_TMA, tma)
            outs.append(g.run(1, T, T.clone(), C, 1.0, dt, *dd).cpu().numpy()[0])
        assert g.device_status() == 0
    assert np.array_equal(outs[0].view(np.int64), outs[1].view(np.int64))
    # the emulated paths' bound is a few ulps of the largest value (2^-52) and
    # 2^-44 of Ci sum |w d2| <= 12 / 6.1 < 2; the reference's own roundings are
    # far below that
    assert np.abs(outs[0] - ref).max() <= 2.0 ** -42
