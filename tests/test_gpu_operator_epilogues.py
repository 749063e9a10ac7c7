"""The operator's epilogues in every launch variant: the Chebyshev step in all storages, and the
two of the CG (NORM: out = Q in and the shares of |out|^2; RESID: out = y - alpha Q in, in place,
and the shares), against the FP64 oracle and, bit for bit, against each other.

The lattices' sites fill no block (1080, 3000 and 24 physical sites) and the vectors no group of 2
or 4.  Tolerances, max-norm relative to the largest output component: 1e-5 for FP32 storage (as
for the plain operator), for 16-bit storage the plain operator's.  Sums of shares against the FP64
sum of the stored outputs' squares: 1e-5 (48 squares in an FP32 chain at most, each addition
2^-24, then a sum to 2^-40).
"""
import numpy as np
import pytest

from oracle.dirac import WilsonDirac
from synth_inputs import make_config, random_spinor

pytestmark = pytest.mark.gpu
F32, CANON, F16, BF16 = 0, 1, 2, 3
CHEB, NORM, RESID = 1, 2, 3
SHAPES = [(6, 5, 0b111, True, 7), (10, 3, 0b011, False, 5), (2, 3, 0b001, False, 6), (4, 4, 0b111, False, 1)]
M0 = 0.07
C, S1, S2 = 3.7, 0.31, 0.77


@pytest.fixture(scope="module")
def lib():
    import internals
    return internals.load()


def problem(shape):
    import torch
    import paper_2108_11989_gb300 as qs
    L, T, mask, anti, n = shape
    cfg = make_config(T=T, L=L, eps=0.6, theta_sigma=0.4, csw_su3=1.9, csw_u1=1.0, seed=3, cstar_mask=mask,
                      t_antiperiodic=anti)
    lat = qs.Lattice(L, T, mask, anti)
    lat.load_gauge(cfg.su3, cfg.theta, cfg.csw_su3, cfg.csw_u1)
    v = [random_spinor(7 + i, T, L, n).astype(np.complex64).astype(np.complex128).reshape(n, -1) for i in range(3)]
    dev = [torch.from_numpy(a.copy().view(np.float64)).float().cuda().reshape(-1) for a in v]
    torch.cuda.synchronize()
    return qs, lat, cfg, n, v, dev


def host(t, n):
    return t.double().cpu().numpy().reshape(n, -1).view(np.complex128)


def ptr(t):
    return None if t is None else t.data_ptr()


def call(lib, lat, variant, storage, epi, n, x, out, y=None, xo=None, alpha=None, live=None, part=None):
    import torch
    torch.cuda.synchronize()
    s = lib.t_d32(lat.h, variant, storage, epi, n, M0, ptr(x), ptr(out), ptr(y), ptr(xo), C, S1, S2, ptr(alpha), ptr(live),
                  ptr(part))
    assert s == 0


@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_norm_and_resid(lib, shape):
    import torch
    qs, lat, cfg, n, v, dev = problem(shape)
    ns, nt = cfg.n_sites, lib.t_ntile(lat.h)
    op = WilsonDirac(cfg)
    Q = np.stack([op.apply_Q(v[0][r], M0) for r in range(n)])
    al = np.linspace(-0.8, 1.3, n).astype(np.float32)
    R = v[1] - al[:, None].astype(np.float64) * Q
    x, y = [qs.to_tiled(t, ns) for t in dev[:2]]
    alpha = torch.from_numpy(al).cuda()
    mask = [r % 3 != 1 for r in range(n)]
    masks = {"all": None, "some": torch.tensor(mask, dtype=torch.int32, device="cuda")}
    first = {}
    for variant in range(lib.t_nvariants()):
        for name, live in masks.items():
            on = [True] * n if live is None else mask
            for epi, ref in ((NORM, Q), (RESID, R)):
                out = torch.full_like(x, 3.0) if epi == NORM else y.clone()
                before = out.clone()
                part = torch.full((n, nt), -1.0, dtype=torch.float64, device="cuda")
                call(lib, lat, variant, F32, epi, n, x, out, y=out if epi == RESID else None, alpha=alpha, live=live,
                     part=part)
                got = host(qs.from_tiled(out, ns), n)
                sums, o = part.sum(1).cpu().numpy(), out.reshape(n, -1)
                for r in range(n):
                    if not on[r]:
                        assert torch.equal(o[r], before.reshape(n, -1)[r]) and bool((part[r] == -1.0).all())
                        continue
                    assert np.abs(got[r] - ref[r]).max() <= 1e-5 * np.abs(ref[r]).max(), (variant, epi, r)
                    want = float((o[r].double() ** 2).sum())
                    assert abs(sums[r] - want) <= 1e-5 * want, (variant, epi, r)
                f = first.setdefault((name, epi), (out, part))
                assert torch.equal(out, f[0]), (variant, epi, name)
                assert torch.equal(part, f[1]), (variant, epi, name)
    lat.close()


@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_chebyshev_step(lib, shape):
    import torch
    from test_gpu_dslash import TOL16, pack16
    qs, lat, cfg, n, v, dev = problem(shape)
    ns = cfg.n_sites
    op = WilsonDirac(cfg)
    for storage in (F32, CANON, F16, BF16):
        if storage in (F16, BF16):
            p, tol, prec = ("f16", TOL16["f16"], qs.QS_F16) if storage == F16 else ("bf16", TOL16["bf16"], qs.QS_BF16)
            packed = [pack16(a.reshape(n, ns, 12), p) for a in v]
            t = [b.cuda() if torch.is_tensor(b) else torch.from_numpy(b).cuda() for b, _ in packed]
            w = [rep.reshape(n, -1) for _, rep in packed]
        else:
            tol, w = 1e-5, v
            t = [qs.to_tiled(d, ns) if storage == F32 else d for d in dev]
        ref = np.stack([S1 * (op.apply_Q(w[0][r], M0) - C * w[1][r]) - S2 * w[2][r] for r in range(n)])
        first = None
        for variant in range(lib.t_nvariants()):
            out = torch.zeros_like(t[0])
            call(lib, lat, variant, storage, CHEB, n, t[0], out, y=t[1], xo=t[2])
            if first is None:
                first = out
                if storage in (F16, BF16):
                    e = torch.empty(n * ns * 24, dtype=torch.float32, device="cuda")
                    qs.convert_spinors(lat.h, out, prec, e, qs.QS_F32, n)
                    torch.cuda.synchronize()
                else:
                    e = out
                got = host(e if storage == CANON else qs.from_tiled(e, ns), n)
                assert np.abs(got - ref).max() <= tol * np.abs(ref).max(), storage
            assert torch.equal(out, first), (variant, storage)
    lat.close()


@pytest.mark.parametrize("shape", SHAPES + [(8, 8, 0b111, False, 3)], ids=str)
def test_shares_against_64_bits(lib, shape):
    """The shares' sum against the FP64 sum of the stored outputs' squares to 4e-12: the high parts
    of a site's 24 squares and of a warp's 32 sites are summed without error, and the low parts,
    at most 18 roundings of 2^-24 of the sum, in at most 54 FP32 operations: 972 x 2^-48."""
    import torch
    qs, lat, cfg, n, v, dev = problem(shape)
    ns, nt = cfg.n_sites, lib.t_ntile(lat.h)
    x, y = [qs.to_tiled(t, ns) for t in dev[:2]]
    alpha = torch.linspace(-0.8, 1.3, n, device="cuda")
    for variant in (1, 5):
        for epi in (NORM, RESID):
            out = y.clone()
            part = torch.zeros((n, nt), dtype=torch.float64, device="cuda")
            call(lib, lat, variant, F32, epi, n, x, out, y=out if epi == RESID else None, alpha=alpha, part=part)
            want = (out.reshape(n, -1).double() ** 2).sum(1)
            assert bool(((part.sum(1) - want).abs() <= 4e-12 * want).all()), (variant, epi, (part.sum(1) / want - 1).tolist())
    lat.close()


@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_plain_in_every_storage(lib, shape):
    """The plain operator in all storages, BF16 among them: every variant gives the same bits, and
    the oracle's values to the tolerances above."""
    import torch
    from test_gpu_dslash import TOL16, pack16
    qs, lat, cfg, n, v, dev = problem(shape)
    ns = cfg.n_sites
    op = WilsonDirac(cfg)
    for storage, kind in ((F32, None), (CANON, None), (F16, "f16"), (BF16, "bf16")):
        if kind:
            buf, rep = pack16(v[0].reshape(n, ns, 12), kind)
            x, w, tol = torch.from_numpy(buf).cuda(), rep.reshape(n, -1), TOL16[kind]
        else:
            x, w, tol = qs.to_tiled(dev[0], ns) if storage == F32 else dev[0], v[0], 1e-5
        ref = np.stack([op.apply_Q(w[r], M0) for r in range(n)])
        outs = []
        for variant in range(lib.t_nvariants()):
            outs.append(torch.zeros_like(x))
            call(lib, lat, variant, storage, 0, n, x, outs[-1])
            assert torch.equal(outs[-1], outs[0]), (variant, storage)
        e = outs[0]
        if kind:
            e = torch.empty(n * ns * 24, dtype=torch.float32, device="cuda")
            qs.convert_spinors(lat.h, outs[0], qs.QS_F16 if storage == F16 else qs.QS_BF16, e, qs.QS_F32, n)
            torch.cuda.synchronize()
        got = host(e if storage == CANON else qs.from_tiled(e, ns), n)
        assert np.abs(got - ref).max() <= tol * np.abs(ref).max(), storage
    lat.close()
