"""A mass that is not a number, or so large that Q^2 leaves the number range, ends the
eigensolver with a status (QS_ENOCONV: its dense eigensolver cannot converge), and the handle
and the GPU context go on working."""
import numpy as np
import pytest

from synth_inputs import make_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["QS_F64", "QS_F32", "QS_F16", "QS_BF16"])
@pytest.mark.parametrize("k", [2, 8, 64])
def test_nonfinite_mass_is_a_status(prec, k):
    import paper_2108_11989_gb300 as qs
    cfg = make_config(T=4, L=2, eps=0.5, theta_sigma=0.3, csw_su3=1.5, csw_u1=1.0, seed=1)
    lat = qs.Lattice(cfg.L, cfg.T)
    lat.load_gauge(cfg.su3, cfg.theta, cfg.csw_su3, cfg.csw_u1)
    eig = dict(k=k, nwant=2, tol=1e-6, precision=getattr(qs, prec))
    for m0 in (float("nan"), float("inf"), -float("inf")):
        with pytest.raises(qs.QStarError) as e:
            lat.lowmodes_at_mass(m0, qs.eig_default_opts(**eig))
        assert e.value.code == -4, m0
        if k >= 4:
            with pytest.raises(qs.QStarError) as e:
                lat.pfaffian_sign(m0, qs.sign_default_opts(eig=eig))
            assert e.value.code == -4 and e.value.report["fail_reason"] == 1, m0
    ev, _, st = lat.lowmodes_at_mass(-0.2, qs.eig_default_opts(**dict(eig, k=16, precision=qs.QS_F32)))
    assert np.isfinite(ev).all() and st["iterations"] >= 0
    lat.close()
