"""Operator products between compact vectors in one kernel (gkb_apply,
gkb_apply_noalloc): against the oracle's sparse matrices at sizes around the
kernel's tiles (32 x 16 positions in 2D, 32 x 8 x 8 in 3D), with natural sides,
and with the result written over the input, which goes through the padded
arrays and must give the same bits."""
import numpy as np
import pytest

from gpu_helpers import make_handle, oracle_problem

pytestmark = pytest.mark.gpu

D, N = 0, 1


@pytest.mark.parametrize("n,bc", [((31, 15), (D, D, D, D)), ((32, 16), (D, N, N, D)), ((33, 17), (N, D, D, N)),
                                  ((2, 3), (D, D, D, D)), ((31, 7, 8), (D,) * 6), ((32, 8, 7), (D, N, N, D, N, D)),
                                  ((33, 9, 17), (N, D, D, N, D, N)), ((2, 2, 2), (D,) * 6)])
def test_products_match_oracle_and_in_place(lib, n, bc):
    import torch
    gk = lib
    gamma = 37.0
    grid, ops = oracle_problem(n, bc, 1.3, gamma)
    h = make_handle(gk, n, bc, 1.3, gamma, inner=0)
    try:
        rng = np.random.default_rng(11)
        for op, mat in ((gk.GKB_OP_W, ops["W"]), (gk.GKB_OP_M, ops["M"]), (gk.GKB_OP_A, ops["A"]),
                        (gk.GKB_OP_AT, ops["A"].T.tocsr())):
            x = rng.standard_normal(mat.shape[1])
            ref = mat @ x
            buf = torch.zeros(max(mat.shape), dtype=torch.float64, device="cuda")
            buf[:len(x)] = torch.tensor(x)
            y = torch.full((len(ref),), float("nan"), dtype=torch.float64, device="cuda")
            gk.gkb_apply(h, op, buf[:len(x)], y)
            # a row sums at most 20 products of O(1) terms of its own scale
            assert np.abs(y.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()
            z = torch.full_like(y, float("nan"))
            s = torch.cuda.current_stream().cuda_stream
            assert gk.gkb_apply_noalloc(gk.make_grid(n, 1.0 / n[0], bc), 1.3, gamma, 0.0, op, buf[:len(x)], z, s) == 0
            assert torch.equal(y, z)
            gk.gkb_apply(h, op, buf[:len(x)], buf[:len(ref)])
            assert torch.equal(buf[:len(ref)], y)
    finally:
        gk.gkb_destroy(h)
