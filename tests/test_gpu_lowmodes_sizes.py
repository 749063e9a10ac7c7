"""Low eigenvalues at block sizes and volumes that fill no tile of the solver's kernels, against
the dense oracle.

2^3 x 3 (1152 reals per vector: one reduction block, 576 complex entries: a ragged last chunk of
the Gram kernels) and 4^3 x 2, blocks of 4 to 48 vectors (Gram and rotation tiles are 4 wide, the
Jacobi rounds pair k / 2 columns).  Tolerance: 1e-10 relative on the wanted eigenvalues, which
converge to a residual of 1e-9 (their error is of second order in it).
"""
import numpy as np
import pytest

from oracle.dirac import WilsonDirac
from synth_inputs import make_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("L,T,k", [(2, 3, 4), (2, 3, 10), (2, 3, 26), (2, 3, 48), (4, 2, 14), (4, 2, 34)])
def test_block_sizes_against_dense(L, T, k, precision):
    import paper_2108_11989_gb300 as qs
    cfg = make_config(T=T, L=L, eps=0.9, theta_sigma=0.4, csw_su3=1.3, csw_u1=0.8, seed=21 + L)
    lat = qs.Lattice(L, T)
    lat.load_gauge(cfg.su3, cfg.theta, cfg.csw_su3, cfg.csw_u1)
    m0 = 0.1
    ev, rs, _ = lat.lowmodes_at_mass(m0, qs.eig_default_opts(k=k, nwant=2, tol=1e-9, cheb_degree=24, max_iter=600,
                                                             warm_start=0, precision=precision))
    ref = np.linalg.eigvalsh(WilsonDirac(cfg).dense_Q(m0))
    ref = ref[np.argsort(np.abs(ref), kind="stable")]
    assert np.allclose(np.sort(np.abs(ev[:2])), np.abs(ref[:2]), rtol=1e-10, atol=1e-14), (ev[:2], ref[:4])
    for i in range(2):
        assert np.abs(ref - ev[i]).min() <= rs[i] + 1e-12
    lat.close()
