"""The operator first met inside a graph capture, where its variants cannot be timed: the thread per
site on problems up to 32768 physical sites x vectors, and the same bits as a timed call."""
import pytest

from synth_inputs import make_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,T,nrhs", [(2, 3, 1), (6, 5, 7), (8, 8, 8), (8, 8, 9)])
def test_first_call_in_a_capture(L, T, nrhs):
    import torch
    import internals
    import paper_2108_11989_gb300 as qs
    cfg = make_config(T=T, L=L, eps=0.6, theta_sigma=0.4, csw_su3=1.9, csw_u1=1.0, seed=3)
    st = torch.cuda.Stream()
    lat = qs.Lattice(L, T, stream=st)
    lat.load_gauge(cfg.su3, cfg.theta, cfg.csw_su3, cfg.csw_u1)
    assert internals.load().t_fixed_variant(lat.h, nrhs) == (5 if L ** 3 * T * nrhs <= 32768 else 1)
    x = torch.randn(nrhs * lat.n_sites * 24, device="cuda")
    y, ref = torch.zeros_like(x), torch.zeros_like(x)
    torch.cuda.synchronize()
    with torch.cuda.stream(st):   # another number of vectors first: the kernels are loaded
        lat.apply_Q(0.1, x[: lat.n_sites * 24].repeat(nrhs + 30), torch.zeros((nrhs + 30) * lat.n_sites * 24, device="cuda"))
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            lat.apply_Q(0.1, x, y)
        g.replay()
        torch.cuda.synchronize()
    other = qs.Lattice(L, T, stream=st)
    other.load_gauge(cfg.su3, cfg.theta, cfg.csw_su3, cfg.csw_u1)
    other.apply_Q(0.1, x, ref)
    torch.cuda.synchronize()
    assert torch.equal(y, ref)
    other.close()
    lat.close()
