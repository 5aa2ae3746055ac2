"""The bounds-checked build (test_gpu_bounds_check) on grids whose stencils run
as stencil and fix-up launches and as the row-copy kernel."""
import numpy as np
import pytest

import test_gpu_bounds_check as base

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dims", [((130, 130, 70), (1, 1, 1)), ((67, 21, 19), (2, 2, 2))])
def test_checked_build_same_bits_no_failed_test(n, dims, tmp_path, monkeypatch):
    monkeypatch.setattr(base, "SCRIPT", base.SCRIPT.replace("(70, 21, 19), (2, 2, 2)", f"{n}, {dims}"))
    assert f"{n}, {dims}" in base.SCRIPT
    from paper_2211_15716_gb300 import build
    build.build()
    build.build(checked=True)
    rel, f0, s0 = base._run(tmp_path, False)
    chk, f1, s1 = base._run(tmp_path, True)
    assert (f0, f1, s0, s1) == (0, 1, 0, 0)
    assert np.array_equal(rel.view(np.uint64), chk.view(np.uint64))
