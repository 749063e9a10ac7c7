"""The Rayleigh-Ritz matrix V^H Q V of the FP32 stage against 64 bits: both triangles are computed, each
with errors of its own, so that their mean, which the dense eigensolver takes, has a smaller error
than one of them (by a factor of 0.71 for independent errors; 0.85 allows for 192 samples)."""
import numpy as np
import pytest

from synth_inputs import make_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,T,k", [(4, 6, 16), (6, 4, 22), (8, 8, 32)])
def test_mean_of_both_triangles(L, T, k):
    import torch
    import internals
    import paper_2108_11989_gb300 as qs
    cfg = make_config(T=T, L=L, eps=0.5, theta_sigma=0.3, csw_su3=1.5, csw_u1=1.0, seed=4)
    lat = qs.Lattice(L, T)
    lat.load_gauge(cfg.su3, cfg.theta, cfg.csw_su3, cfg.csw_u1)
    g = torch.Generator(device="cuda")
    g.manual_seed(k)
    v = torch.randn((k, cfg.n_sites * 12, 2), dtype=torch.float64, device="cuda", generator=g)
    V = torch.linalg.qr(torch.view_as_complex(v).T)[0].T.contiguous()
    V32 = torch.view_as_real(V).float().contiguous()
    QV = torch.empty_like(V32)
    H = np.zeros((k, k), dtype=np.complex128)
    torch.cuda.synchronize()
    assert internals.load().t_rr32(lat.h, k, -0.2, V32.data_ptr(), QV.data_ptr(), H.ctypes.data) == 0
    a, b = [torch.view_as_complex(t.double()) for t in (V32, QV)]
    G = (a.conj() @ b.T).cpu().numpy()
    assert np.abs(H - G).max() <= 1e-5 * np.abs(G).max()
    want = (G + G.conj().T) / 2
    i, j = np.triu_indices(k, 1)
    off = i // 4 != j // 4
    i, j = i[off], j[off]
    rms = lambda e: np.sqrt(np.mean(np.abs(e) ** 2))  # noqa: E731
    one = rms(H[i, j] - want[i, j])
    mean = rms((H + H.conj().T)[i, j] / 2 - want[i, j])
    assert mean <= 0.85 * one, (mean, one)
    lat.close()
