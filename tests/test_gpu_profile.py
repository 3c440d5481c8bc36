"""A profiled solve can time the launches that a solve without profiling makes
(profile = 2): the same number of them in every class, all timed. With
profile = 1 the steps of a 2D V-cycle are launched one by one."""
import numpy as np
import pytest

from gpu_helpers import gpu_solve, make_handle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,prec,var", [((64, 48), 0, 0), ((192, 160), 1, 0), ((96, 64), 1, 1), ((16, 16, 16), 1, 0)])
def test_profile_of_the_launches_of_a_solve(lib, n, prec, var):
    gk = lib
    mu = np.exp(0.3 * np.random.default_rng(2).standard_normal(n)) if var else 1.0
    got = {}
    for profile in (0, 1, 2):
        h = make_handle(gk, n, (0,) * (2 * len(n)), mu, 10.0, precision=prec, use_graph=0, profile=profile)
        try:
            m, nc = gk.gkb_layout(h)
            rc, w, p = gpu_solve(gk, h, np.random.default_rng(3).standard_normal(m), np.zeros(nc))
            assert rc == gk.GKB_OK, gk.gkb_last_error(h)
            got[profile] = (w, p, gk.gkb_stats(h))
        finally:
            gk.gkb_destroy(h)
    for profile in (1, 2):
        assert np.array_equal(got[0][0], got[profile][0]) and np.array_equal(got[0][1], got[profile][1])
    ran, steps, timed = (got[k][2] for k in (0, 1, 2))
    assert timed["kernel_launches"] == ran["kernel_launches"]
    for k, count in timed["kernel_launches"].items():
        assert (timed["kernel_ms"][k] > 0) == (count > 0), k
    fused = len(n) == 2
    assert (sum(steps["kernel_launches"].values()) > sum(ran["kernel_launches"].values())) == fused


@pytest.mark.parametrize("prec", [0, 1])
def test_profiled_handles_tune_the_same_launches(lib, prec):
    """A profiled handle's choice is the cached one of every other handle of its
    key, so it is made with the launches of a solve without profiling. A grid
    and its transposed (another key, the same work) are timed within 40 % of
    each other; with separate launches the profiled one took twice as long."""
    import torch
    gk = lib
    ms = []
    for n, profile in (((112, 80), 1), ((80, 112), 0)):
        opt = gk.gkb_default_options()
        opt.precision = prec
        opt.autotune = 1
        opt.profile = profile
        opt.stream = torch.cuda.current_stream().cuda_stream
        h = gk.gkb_create(opt)
        try:
            gk.gkb_set_problem(h, gk.make_grid(n, 1.0 / n[0], (0,) * 4), None, 1.0, 30.0, 0.0)
            ms.append(gk.gkb_stats(h)["tuned_inner_ms"])
        finally:
            gk.gkb_destroy(h)
    assert 1 / 1.4 <= ms[0] / ms[1] <= 1.4, ms
