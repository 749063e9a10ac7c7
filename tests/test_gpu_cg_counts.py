"""The inner CG of the eigensolver on vectors that converge at different iterations: the same
solutions, bit for bit, as each vector alone; and counters (operator applications, iterations,
profiled bytes) that hold the work done, not the vectors and launches skipped after convergence."""
import ctypes

import numpy as np
import pytest

from synth_inputs import make_config

pytestmark = pytest.mark.gpu
M0 = -0.1


@pytest.fixture(scope="module")
def problem():
    import torch
    import internals
    import paper_2108_11989_gb300 as qs
    cfg = make_config(T=6, L=4, eps=0.5, theta_sigma=0.3, csw_su3=1.5, csw_u1=1.0, seed=2)
    lat = qs.Lattice(cfg.L, cfg.T)
    lat.load_gauge(cfg.su3, cfg.theta, cfg.csw_su3, cfg.csw_u1)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    b = torch.randn((4, cfg.n_sites * 24), device="cuda", generator=g)
    for _ in range(8):   # vector 1 loses its low modes and converges early
        y = torch.empty_like(b[1])
        lat.apply_Q(M0, b[1], y, tiled=True)
        b[1] = y / y.norm()
    b[2] = 0
    torch.cuda.synchronize()
    yield internals.load(), lat, cfg, b
    lat.close()


def cg(lib, lat, b, tol, cap):
    import torch
    b = b.contiguous()
    x = torch.full_like(b, float("nan"))
    n = (ctypes.c_int64 * 3)()
    torch.cuda.synchronize()
    assert lib.t_cg(lat.h, b.shape[0], M0, tol, cap, b.data_ptr(), x.data_ptr(), n) == 0
    return x, list(n)


@pytest.mark.parametrize("cap", [5000, 40, 7, 1])
def test_counts_are_of_work_done(problem, cap):
    import torch
    lib, lat, cfg, b = problem
    tol = 1e-4
    alone = [cg(lib, lat, b[r:r + 1], tol, cap) for r in range(4)]
    its = [n[2] for _, n in alone]
    assert its[2] == 0 and its[0] > 0 and max(its) <= cap
    if cap == 5000:
        assert its[1] < its[0] < cap
        q = torch.empty_like(b[:1])
        t = torch.empty_like(b[:1])
        lat.apply_Q(M0, alone[0][0], t, tiled=True)
        lat.apply_Q(M0, t, q, tiled=True)
        assert (q - b[:1]).norm() <= 3 * tol * b[:1].norm()
    cg(lib, lat, b, tol, cap)   # the operator's variant is timed here
    lat.set_profiling(True)
    x, n = cg(lib, lat, b, tol, cap)
    prof = lat.get_profile()
    lat.set_profiling(False)
    for r in range(4):
        assert torch.equal(x[r], alone[r][0][0]), r
    assert n == [2 * sum(its), max(its), max(its)]
    f32 = prof["f32"]
    assert f32["bytes"] == cfg.n_sites * (5 * 96 * sum(its) + 2 * 288 * max(its))
    assert f32["launches"] >= 2 * max(its)


def test_zero_vectors_do_no_work(problem):
    lib, lat, _, b = problem
    x, n = cg(lib, lat, b[2:3].repeat(2, 1), 1e-4, 100)
    assert n == [0, 0, 0] and bool((x == 0).all())
