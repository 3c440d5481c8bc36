"""The fused V-cycle legs (one kernel for a 2D level's down half, one for its up
half) against the separate launches of the same steps, which a profiled handle
takes: the legs form every value by the same operations in the same order, so
one V-cycle must agree bit for bit. Sizes around the tiles' edges (8 cells; 22
and 54 cells of a 32 and a 64 wide tile with its halo), levels of a few cells,
ragged sides, every smoother degree that has an instance."""
import numpy as np
import pytest

from gpu_helpers import make_handle

pytestmark = pytest.mark.gpu

FP64, MIXED = 0, 1


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("n,prec,var", [((16, 12), FP64, 0), ((72, 40), FP64, 0), ((136, 120), FP64, 0),
                                        ((12, 20), MIXED, 0), ((44, 66), MIXED, 0), ((108, 112), MIXED, 0),
                                        ((248, 56), MIXED, 0), ((12, 10), MIXED, 1), ((44, 64), MIXED, 1),
                                        ((92, 152), MIXED, 1)])
def test_legs_equal_separate_launches(lib, n, prec, var, degree):
    gk = lib
    mu = np.exp(0.7 * np.random.default_rng(5).standard_normal(n)) if var else 1.0
    out = []
    for profile in (0, 1):
        h = make_handle(gk, n, (0,) * 4, mu, 200.0, precision=prec, degree=degree, profile=profile)
        try:
            m, _ = gk.gkb_layout(h)
            z = np.empty(m)
            gk.gkb_precond(h, np.random.default_rng(6).standard_normal(m), z)
            out.append(z)
        finally:
            gk.gkb_destroy(h)
    assert np.all(np.isfinite(out[0])) and np.any(out[0])
    assert np.array_equal(out[0], out[1])
