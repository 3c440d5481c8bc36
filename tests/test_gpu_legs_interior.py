"""The instances of the fused V-cycle legs for tiles away from the sides,
against the separate launches of the same steps (a handle with profile = 1), bit
for bit, at every smoother degree. A tile of a leg takes them when the blocks
of 32 x 8 positions around it, halo included, lie three positions inside the
level; `inner_tiles` counts those, so that a size does reach them."""
import numpy as np
import pytest

from gpu_helpers import make_handle

pytestmark = pytest.mark.gpu

FP64, MIXED = 0, 1


def inner_tiles(n, degree, down, ew, eh):
    """Tiles of ew x eh positions, halo included, that are wholly interior."""
    lo, hi = 2 * degree + (2 if down else 0), 2 * degree
    count = 0
    for e0 in range(-lo, n[0] - lo, ew - lo - hi):
        for e1 in range(-lo, n[1] - lo, eh - lo - hi):
            ok = e0 >= 0 and e1 >= 0
            for i, j in ((e0, e1), (e0 + ew - 1, e1 + eh - 1)):
                a, b = i & ~31, j & ~7
                ok = ok and a >= 3 and a + 31 <= n[0] - 3 and b >= 3 and b + 7 <= n[1] - 3
            count += ok
    return count


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("n,prec,var", [((136, 72), MIXED, 0), ((200, 136), MIXED, 0), ((104, 72), MIXED, 1),
                                        ((168, 104), MIXED, 1), ((128, 120), FP64, 0)])
def test_interior_tiles(lib, n, prec, var, degree):
    gk = lib
    for down in (0, 1):
        halo = 4 * degree + (2 if down else 0)
        ew, eh = (8 + halo, 8 + halo) if prec == FP64 else (32, 32) if var else (64, 32)
        assert inner_tiles(n, degree, down, ew, eh) > 0
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
