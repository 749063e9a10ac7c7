"""qs_solve_D on right-hand sides that differ: one zero, one that converges early and one that takes
long give, bit for bit, what each gives alone, and the count is the longest; a right-hand side with a
NaN is QS_ENUMERIC, and the others are solved all the same."""
import numpy as np
import pytest

from synth_inputs import make_config, random_spinor

pytestmark = pytest.mark.gpu
M0, TOL = -0.2, 1e-10


@pytest.fixture(scope="module", params=[(6, 4), (4, 2)], ids=str)
def problem(request):
    import torch
    import paper_2108_11989_gb300 as qs
    T, L = request.param
    cfg = make_config(T=T, L=L, eps=0.6, theta_sigma=0.3, csw_su3=1.5, csw_u1=1.0, seed=6)
    lat = qs.Lattice(L, T)
    lat.load_gauge(cfg.su3, cfg.theta, cfg.csw_su3, cfg.csw_u1)
    b = torch.from_numpy(random_spinor(5, T, L, 3).reshape(3, -1).view(np.float64).copy()).cuda()
    b[0] = 0
    for _ in range(30):   # vector 1 keeps the high modes and converges early
        y = torch.empty_like(b[1])
        lat.apply_Q(M0, b[1], y)
        b[1] = y / y.norm()
    torch.cuda.synchronize()
    yield qs, lat, b
    lat.close()


def solve(lat, b, even_odd):
    import torch
    b = b.contiguous()
    x = torch.full_like(b, float("nan"))
    return x, lat.solve_D(M0, b, x, even_odd=even_odd, tol=TOL)


@pytest.mark.parametrize("even_odd", [True, False])
def test_each_as_alone(problem, even_odd):
    import torch
    qs, lat, b = problem
    alone = [solve(lat, b[r:r + 1], even_odd) for r in range(3)]
    x, n = solve(lat, b, even_odd)
    its = [a[1] for a in alone]
    assert its[0] == 0 and 0 < its[1] < its[2] == n, its
    for r in range(3):
        assert torch.equal(x[r], alone[r][0][0]), r
    assert bool((x[0] == 0).all())


@pytest.mark.parametrize("even_odd", [True, False])
@pytest.mark.parametrize("site", [0, 1])
def test_nan_in_one_right_hand_side(problem, even_odd, site):
    import torch
    qs, lat, b = problem
    clean, _ = solve(lat, b, even_odd)
    bad = b.clone()
    bad[1, 24 * site + 3] = float("nan")
    x = torch.full_like(bad, float("nan"))
    with pytest.raises(qs.QStarError) as e:
        lat.solve_D(M0, bad, x, even_odd=even_odd, tol=TOL)
    assert e.value.code == -6
    assert torch.equal(x[0], clean[0]) and torch.equal(x[2], clean[2])
