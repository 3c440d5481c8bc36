"""Operator products written over their input go through the padded arrays and
the kernels that the solver runs (tiles; box and shell in 3D; above 2^19 cells
the FP64 tile's fast path), with and without a handle: against the oracle's
matrices, and bit for bit the products between separate vectors."""
import numpy as np
import pytest

from gpu_helpers import make_handle, oracle_problem

pytestmark = pytest.mark.gpu

D, N = 0, 1


def _ops(gk, ops):
    return ((gk.GKB_OP_W, ops["W"]), (gk.GKB_OP_M, ops["M"]), (gk.GKB_OP_A, ops["A"]),
            (gk.GKB_OP_AT, ops["A"].T.tocsr()))


@pytest.mark.parametrize("n,bc", [((1024, 1024), (D,) * 4), ((1021, 517), (D, N, N, D)), ((733, 719), (N, D, D, N)),
                                  ((40, 36, 34), (D,) * 6), ((67, 17, 35), (N, D, D, N, D, N)),
                                  ((16, 16, 16), (D, N, D, D, D, D)), ((35, 30, 15), (D,) * 6)])
def test_handle_products_in_place(lib, n, bc):
    import torch
    gk = lib
    _, ops = oracle_problem(n, bc, 1.3, 370.0)
    rng = np.random.default_rng(12)
    for variant in (0, 1, 2):
        h = make_handle(gk, n, bc, 1.3, 370.0, inner=0, kernel_variant=variant)
        try:
            for op, mat in _ops(gk, ops):
                x = rng.standard_normal(mat.shape[1])
                ref = mat @ x
                buf = torch.zeros(max(mat.shape), dtype=torch.float64, device="cuda")
                buf[:len(x)] = torch.tensor(x)
                y = torch.full((len(ref),), float("nan"), dtype=torch.float64, device="cuda")
                gk.gkb_apply(h, op, buf[:len(x)], y)
                gk.gkb_apply(h, op, buf[:len(x)], buf[:len(ref)])
                assert torch.equal(buf[:len(ref)], y), (variant, op)
                # a row sums at most 20 products of terms of its own scale
                assert np.abs(y.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max(), (variant, op)
        finally:
            gk.gkb_destroy(h)


@pytest.mark.parametrize("shift", [0, 3])
def test_products_without_a_handle_in_place(lib, shift):
    """The static work arrays keep what the call before left in them: two
    rounds over grids of several sizes and all operators, the result over the
    input, or `shift` entries on."""
    import torch
    gk = lib
    grids = []
    for n, bc in (((40, 37), (D, N, D, D)), ((64, 64), (D,) * 4), ((3, 2), (N, D, D, D)),
                  ((12, 10, 9), (D, D, N, D, D, N)), ((17, 18, 20), (D,) * 6)):
        grids.append((n, bc, oracle_problem(n, bc, 0.7, 25.0)[1]))
    rng = np.random.default_rng(13)
    s = torch.cuda.current_stream().cuda_stream
    for _ in range(2):
        for n, bc, ops in grids:
            grid = gk.make_grid(n, 1.0 / n[0], bc)
            for op, mat in _ops(gk, ops):
                x = rng.standard_normal(mat.shape[1])
                ref = mat @ x
                buf = torch.zeros(max(mat.shape) + shift, dtype=torch.float64, device="cuda")
                xd = buf[:len(x)]
                xd.copy_(torch.tensor(x))
                y = torch.empty(len(ref), dtype=torch.float64, device="cuda")
                assert gk.gkb_apply_noalloc(grid, 0.7, 25.0, 0.0, op, xd, y, s) == gk.GKB_OK
                out = buf[shift:shift + len(ref)]
                assert gk.gkb_apply_noalloc(grid, 0.7, 25.0, 0.0, op, xd, out, s) == gk.GKB_OK
                assert torch.equal(out, y), (n, op)
                assert np.abs(y.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max(), (n, op)
