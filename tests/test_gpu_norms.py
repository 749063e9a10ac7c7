"""Norms of block vectors: a vector's norm is the same, bit for bit, alone and in a block of any
size (through the public allocation-free entry, whose output is the same in both)."""
import numpy as np
import pytest

from synth_inputs import make_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("L,T", [(2, 3), (4, 6), (8, 8), (12, 12)])
def test_norm_does_not_depend_on_the_block(L, T, dtype):
    import torch
    import paper_2108_11989_gb300 as qs
    cfg = make_config(T=T, L=L, eps=0.4, theta_sigma=0.3, csw_su3=1.9, csw_u1=1.0, seed=5)
    lat = qs.Lattice(L, T)
    lat.load_gauge(cfg.su3, cfg.theta, cfg.csw_su3, cfg.csw_u1)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    x = torch.randn((64, cfg.n_sites * 24), dtype=getattr(torch, dtype), device="cuda", generator=g)
    norms = {}
    for n in (1, 3, 16, 64):
        out = torch.empty_like(x[:n])
        nrm = torch.empty(n, dtype=torch.float64, device="cuda")
        qs.apply_Q_norm2_noalloc(lat.h, -0.1, x[:n], out, nrm)
        torch.cuda.synchronize()
        norms[n] = nrm.cpu().numpy()
        want = (out.double() ** 2).sum(1).cpu().numpy()
        assert np.all(np.abs(norms[n] - want) <= 1e-6 * want)
    for n in (1, 3, 16):
        assert np.array_equal(norms[n], norms[64][:n]), (n, norms[n] / norms[64][:n] - 1)
    lat.close()


def sums(v, theta=None, b=None):
    """|v_r|^2, or |v_r - theta_r b_r|^2, of FP32 vectors by the solver's reductions."""
    import torch
    import internals
    import paper_2108_11989_gb300 as qs
    lib, lat = internals.load(), qs.Lattice(2, 2)
    k, nr = v.shape
    part = torch.full((k, 608), float("nan"), dtype=torch.float64, device="cuda")
    out = torch.full((k,), float("nan"), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    if b is None:
        s = lib.t_norm2(lat.h, 0, v.data_ptr(), k, nr, part.data_ptr(), out.data_ptr())
    else:
        s = lib.t_resid2(lat.h, v.data_ptr(), b.data_ptr(), theta.data_ptr(), k, nr, part.data_ptr(), out.data_ptr())
    assert s == 0
    lat.close()
    return out.cpu().numpy()


def test_sum_beyond_the_range_is_infinite():
    """Squares whose FP32 sum overflows: infinity (which the solver reports), never NaN (whose square
    root it would take for a zero residual)."""
    import torch
    v = torch.zeros((3, 4608), device="cuda")
    v[1] = 1.5e19          # each square is a number, their sums are not
    v[2, 17] = 1e30
    zero, theta = torch.zeros_like(v), torch.zeros(3, dtype=torch.float64, device="cuda")
    for got in (sums(v), sums(v, theta, zero)):
        assert got[0] == 0 and np.isposinf(got[1:]).all(), got


@pytest.mark.parametrize("L,T", [(2, 3), (4, 4), (4, 8), (6, 8), (8, 12)])
def test_fp32_sums_against_64_bits(L, T):
    """FP32 vectors' norms and residuals to 3e-12 of the FP64 sum of the same squares: a thread adds
    at most 16 squares, the high parts without error, the low parts (16 x 2^-24 of the sum at most)
    in 48 FP32 operations: 768 x 2^-48; the threads' sums are added in FP64."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(L * T)
    v = torch.randn((4, 2 * L ** 3 * T * 24), device="cuda", generator=g)
    b = torch.randn(v.shape, device="cuda", generator=g)
    want = (v.double() ** 2).sum(1).cpu().numpy()
    got = sums(v)
    assert np.all(np.abs(got - want) <= 3e-12 * want), got / want - 1
    theta = torch.tensor([0.0, 1.0, 0.5, -2.0], dtype=torch.float64, device="cuda")
    d = (v.double() - theta[:, None] * b.double()).float()   # one rounding, as a fused multiply-add has
    want = (d.double() ** 2).sum(1).cpu().numpy()
    got = sums(v, theta, b)
    assert np.all(np.abs(got - want) <= 3e-12 * want), got / want - 1
