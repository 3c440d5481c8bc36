"""The single-kernel CG with its vectors on chip (unpreconditioned FP64
problems of at most 12 800 padded unknowns): whole solves against the oracle's,
with natural sides, ragged and tiny sizes (blocks of the cluster without
unknowns), 3D, variable viscosity and a diagonal N."""
import numpy as np
import pytest

from gpu_helpers import energy_rel, gpu_solve, make_handle, oracle_problem, oracle_truth

pytestmark = pytest.mark.gpu

D, N = 0, 1


@pytest.mark.parametrize("n,bc,kind", [((2, 2), (D, D, D, N), "const"), ((5, 3), (D,) * 4, "const"),
                                       ((33, 21), (D, N, N, D), "const"), ((62, 60), (D, N, D, D), "const"),
                                       ((17, 30), (D, N, D, D), "var"), ((20, 18), (D, D, N, D), "ndiag"),
                                       ((5, 4, 6), (D, N, D, D, D, D), "const"), ((9, 8, 7), (N, D, D, D, D, N), "var")])
def test_small_cg_solves_match_oracle(lib, n, bc, kind):
    gk = lib
    rng = np.random.default_rng(4)
    mu = np.exp(0.5 * rng.standard_normal(n)) if kind != "const" else 1.0
    nd = (1.0 / n[0]) ** len(n) * np.exp(0.5 * rng.standard_normal(n)) if kind == "ndiag" else None
    kw = {"n_diag": nd} if nd is not None else {}
    grid, ops = oracle_problem(n, bc, mu, 20.0, **kw)
    g = rng.standard_normal(grid.m)
    r = np.zeros(grid.n_cells)
    ref = oracle_truth(grid, ops, g, r)
    h = make_handle(gk, n, bc, mu, 20.0, inner=0, tol_inner=1e-12, maxit_inner=20000, n_diag=nd)
    try:
        rc, w, p = gpu_solve(gk, h, g, r)
        assert rc == gk.GKB_OK, gk.gkb_last_error(h)
    finally:
        gk.gkb_destroy(h)
    assert energy_rel(ops["M"], w, ref["w"]) <= 1e-8
    assert np.abs(p - ref["p"]).max() <= 1e-6 * max(np.abs(ref["p"]).max(), 1e-300)
