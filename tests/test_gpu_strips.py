"""The operator product with its inner product in column strips, which the CG of
large 2D levels runs on: whole solves leave a first-equation residual that the
separately written products of gkb_apply agree on (one wrong face would leave
1e-3 of it), in as many inner iterations as with the general kernels. Sizes
around a strip's 60 columns and its 1 to 8 rows, narrow grids, odd sizes with
natural sides, variable viscosity."""
import numpy as np
import pytest

from gpu_helpers import gpu_solve, make_handle

pytestmark = pytest.mark.gpu

D, N = 0, 1
FP64, MIXED = 0, 1


@pytest.mark.parametrize("n,bc,prec,var,inner", [
    ((512, 544), (D,) * 4, FP64, 0, 1), ((64, 4160), (D,) * 4, FP64, 0, 1), ((1088, 992), (D,) * 4, FP64, 0, 1),
    ((541, 485), (D, N, N, D), FP64, 0, 0), ((512, 544), (D,) * 4, FP64, 1, 1),
    ((352, 384), (D,) * 4, MIXED, 0, 1), ((64, 2112), (D,) * 4, MIXED, 0, 1), ((992, 1088), (D,) * 4, MIXED, 0, 1),
    ((352, 384), (D,) * 4, MIXED, 1, 1), ((992, 1088), (D,) * 4, MIXED, 1, 1)])
def test_strip_product_solves(lib, n, bc, prec, var, inner):
    gk = lib
    rng = np.random.default_rng(8)
    mu = np.exp(0.3 * rng.standard_normal(n)) if var else 1.0
    iters = []
    for variant in (0, 1):
        h = make_handle(gk, n, bc, mu, 1.0, precision=prec, inner=inner, tol_inner=1e-9, maxit_inner=20000,
                        kernel_variant=variant)
        try:
            m, nc = gk.gkb_layout(h)
            g = np.random.default_rng(9).standard_normal(m)
            rc, w, p = gpu_solve(gk, h, g, np.zeros(nc))
            assert rc == gk.GKB_OK, gk.gkb_last_error(h)
            iters.append(gk.gkb_stats(h)["inner_iterations"])
            if variant == 0:
                Ww, Ap = np.empty(m), np.empty(m)
                gk.gkb_apply(h, gk.GKB_OP_W, w, Ww)
                gk.gkb_apply(h, gk.GKB_OP_A, p, Ap)
                assert np.linalg.norm(g - Ww - Ap) <= 1e-5 * np.linalg.norm(g)
        finally:
            gk.gkb_destroy(h)
    assert abs(iters[0] - iters[1]) <= max(2, 0.03 * iters[1]), iters
