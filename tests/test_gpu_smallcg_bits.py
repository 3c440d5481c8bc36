"""The single-kernel CG with its vectors on chip forms every value by the
operations, in the order, of the general cluster kernel, which kernel_variant 1
runs: whole solves agree bit for bit, over the forms that it takes (2D and 3D,
odd and tiny sizes, up to 12 800 padded unknowns; natural sides; constant and
cell viscosity; diagonal N; no grad-div; an iteration limit that ends the
solve)."""
import numpy as np
import pytest

from gpu_helpers import gpu_solve, make_handle

pytestmark = pytest.mark.gpu

D, N = 0, 1


@pytest.mark.parametrize("n,bc,kind,gamma,maxit", [
    ((2, 2), (D, D, D, N), "const", 20.0, 20000), ((3, 5), (D,) * 4, "const", 0.0, 20000),
    ((31, 33), (D, N, D, D), "const", 100.0, 20000), ((94, 61), (D,) * 4, "const", 20.0, 20000),
    ((62, 97), (N, D, D, N), "const", 20.0, 20000), ((7, 350), (D, D, N, D), "const", 5.0, 20000),
    ((17, 30), (D, N, D, D), "var", 20.0, 20000), ((60, 95), (D,) * 4, "var", 20.0, 20000),
    ((23, 18), (D, D, N, D), "ndiag", 20.0, 20000), ((32, 32), (D, N, D, D), "const", 100.0, 3),
    ((2, 2, 2), (D,) * 6, "const", 20.0, 20000), ((5, 4, 6), (D, N, D, D, D, D), "const", 20.0, 20000),
    ((10, 10, 10), (D,) * 6, "const", 20.0, 20000), ((31, 7, 5), (N, D, D, N, D, D), "const", 20.0, 20000),
    ((9, 8, 7), (N, D, D, D, D, N), "var", 20.0, 20000), ((30, 6, 6), (D,) * 6, "var", 20.0, 20000),
    ((6, 9, 5), (D,) * 6, "ndiag", 20.0, 20000)])
def test_on_chip_and_general_kernel_agree(lib, n, bc, kind, gamma, maxit):
    gk = lib
    rng = np.random.default_rng(4)
    mu = np.exp(0.5 * rng.standard_normal(n)) if kind != "const" else 1.0
    nd = (1.0 / n[0]) ** len(n) * np.exp(0.5 * rng.standard_normal(n)) if kind == "ndiag" else None
    got = []
    for variant in (0, 1):
        h = make_handle(gk, n, bc, mu, gamma, inner=0, tol_inner=1e-11, maxit=40, maxit_inner=maxit, n_diag=nd,
                        kernel_variant=variant)
        try:
            m, nc = gk.gkb_layout(h)
            g = np.random.default_rng(6).standard_normal(m)
            try:
                rc, w, p = gpu_solve(gk, h, g, np.zeros(nc))
            except gk.GkbError as e:
                rc, w, p = e.code, np.zeros(0), np.zeros(0)
            got.append((rc, gk.gkb_stats(h)["inner_iterations"], w, p))
        finally:
            gk.gkb_destroy(h)
    assert got[0][0] == got[1][0] and got[0][1] == got[1][1] > 0
    if maxit == 3:  # the outer limit is reached first and is what the status says
        assert got[0][0] == gk.GKB_ERR_NOT_CONVERGED
    assert np.array_equal(got[0][2], got[1][2]) and np.array_equal(got[0][3], got[1][3])
