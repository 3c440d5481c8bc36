"""Handles and networks on streams that do not wait for the legacy stream:
the work arrays that a call allocates are cleared before its kernels write
them, so the first call at a new size returns the bits of the next one."""
import numpy as np
import pytest

from gpu_helpers import make_handle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h,w", [(1, 8, 8), (2, 64, 96), (4, 260, 292)])
def test_first_training_step_on_its_own_stream(lib, n, h, w):
    import torch
    gk = lib
    st = torch.cuda.Stream()
    x = torch.randn(n, h, w, 3, device="cuda")
    t = torch.randn(n, h, w, 2, device="cuda")
    torch.cuda.synchronize()
    u = gk.gkb_unet_create(3, 16, 32, 2, 7, st.cuda_stream)
    try:
        runs = []
        for _ in range(3):
            g = torch.empty(gk.gkb_unet_num_params(u), dtype=torch.float32, device="cuda")
            torch.cuda.synchronize()
            runs.append((gk.gkb_unet_loss_grad(u, x, t, n, h, w, g), g))
        for loss, g in runs:
            assert loss == runs[-1][0] and torch.equal(g, runs[-1][1]) and bool(g.any())
    finally:
        gk.gkb_unet_destroy(u)


@pytest.mark.parametrize("n,prec", [((64, 48), 0), ((512, 512), 1), ((24, 16, 16), 1)])
def test_solve_set_up_on_its_own_stream(lib, n, prec):
    import torch
    gk = lib
    outs = []
    for st in (torch.cuda.current_stream(), torch.cuda.Stream()):
        with torch.cuda.stream(st):
            h = make_handle(gk, n, (0,) * (2 * len(n)), 1.0, 100.0, precision=prec)
        try:
            m, nc = gk.gkb_layout(h)
            g = np.random.default_rng(3).standard_normal(m)
            w, p = np.empty(m), np.empty(nc)
            gk.gkb_solve(h, g, np.zeros(nc), 1e-8, 5, w, p, None, None)
            outs.append((w, p))
        finally:
            gk.gkb_destroy(h)
    assert np.array_equal(outs[0][0], outs[1][0]) and np.array_equal(outs[0][1], outs[1][1])


def test_networks_of_two_threads(lib):
    """FP32 passes of several networks at once, each from its own thread: a
    launch's shared memory does not depend on another thread's layers."""
    import threading

    import torch
    gk = lib
    n, h, w = 1, 8, 8
    x = torch.randn(n, h, w, 3, device="cuda")
    torch.cuda.synchronize()
    nets = [gk.gkb_unet_create(3, 16, 32, 2, 7, torch.cuda.Stream().cuda_stream) for _ in range(4)]
    ys = [torch.zeros(n, h, w, 2, device="cuda") for _ in nets]
    torch.cuda.synchronize()
    errors = []

    def work(k):
        try:
            for _ in range(400):
                gk.gkb_unet_forward(nets[k], x, n, h, w, ys[k], 0)
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(e)

    try:
        threads = [threading.Thread(target=work, args=(k,)) for k in range(len(nets))]
        for th in threads:
            th.start()
        for th in threads:
            th.join()
        assert not errors, errors
        torch.cuda.synchronize()
        assert bool(ys[0].any()) and all(torch.equal(ys[0], y) for y in ys)
    finally:
        for u in nets:
            gk.gkb_unet_destroy(u)
