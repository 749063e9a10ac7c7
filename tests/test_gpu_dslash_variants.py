"""Every launch variant of the operator against the oracle.

The autotuner picks one variant per shape, so each is forced in turn (a child process with a
tune cache that names it) on lattices whose sites fill no block (6^3 x 5: 1080 physical sites,
10^3 x 3: 3000, 2^3 x 3: 24) and on blocks of vectors that fill no group of 2 or 4.  Tolerances,
max-norm relative to the largest output component: 1e-5 for FP32 storage; for FP16 storage half
a unit in the last place at 1 relative to the site's largest component (2^-11), twice that
allowed; for FP64 1e-13 (about 300 roundings of 2^-53 each on the longest chain, of terms no
larger than the output's scale).
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHAPES = [(6, 5, 0b111, True, [12, 13, 15]), (10, 3, 0b011, False, [5])]
SMALL = [(2, 3, 0b001, False, [1, 3, 6]), (6, 5, 0b111, True, [1, 3, 11]), (4, 4, 0b011, True, [6])]

CHILD = r"""
import sys
sys.path[:0] = [%(root)r, %(root)r + "/tests"]
import numpy as np
import torch
import paper_2108_11989_gb300 as qs
from oracle.dirac import WilsonDirac
from synth_inputs import make_config, random_spinor
from test_gpu_dslash import TOL16, pack16
for L, T, mask, anti, rhs in %(shapes)r:
    cfg = make_config(T=T, L=L, eps=0.6, theta_sigma=0.4, csw_su3=1.9, csw_u1=1.0, seed=3, cstar_mask=mask,
                      t_antiperiodic=anti)
    lat = qs.Lattice(L, T, mask, anti)
    lat.load_gauge(cfg.su3, cfg.theta, cfg.csw_su3, cfg.csw_u1)
    op, ns = WilsonDirac(cfg), cfg.n_sites
    for nrhs in rhs:
        psi = random_spinor(7, T, L, nrhs).astype(np.complex64).astype(np.complex128)
        ref = np.stack([op.apply_Q(psi[r].reshape(-1), 0.07) for r in range(nrhs)]).reshape(nrhs, ns, 12)
        x = torch.from_numpy(np.ascontiguousarray(psi).view(np.float64).copy()).float().cuda().reshape(-1)
        for tiled in (False, True):
            xin = qs.to_tiled(x, ns) if tiled else x
            y = torch.full_like(xin, float("nan"))
            lat.apply_Q(0.07, xin, y, tiled=tiled)
            y = qs.from_tiled(y, ns) if tiled else y
            got = y.double().cpu().numpy().view(np.complex128).reshape(nrhs, ns, 12)
            assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max(), (L, T, nrhs, tiled)
        buf, rep = pack16(psi.reshape(nrhs, ns, 12), "f16")
        ref = np.stack([op.apply_Q(rep[r].reshape(-1), 0.07) for r in range(nrhs)]).reshape(nrhs, ns, 12)
        xb = buf.cuda() if torch.is_tensor(buf) else torch.from_numpy(buf).cuda()
        yb = torch.empty_like(xb)
        lat.apply_Q(0.07, xb, yb, tiled=True, prec=qs.QS_F16)
        y = torch.empty(nrhs * ns * 24, dtype=torch.float32, device="cuda")
        qs.convert_spinors(lat.h, yb, qs.QS_F16, y, qs.QS_F32, nrhs)
        got = qs.from_tiled(y, ns).double().cpu().numpy().view(np.complex128).reshape(nrhs, ns, 12)
        assert np.abs(got - ref).max() <= TOL16["f16"] * np.abs(ref).max(), (L, T, nrhs, "f16")
    lat.close()
"""


@pytest.mark.parametrize("variant", range(7))
def test_forced_variant_matches_oracle(variant, tmp_path):
    import torch
    gpu = torch.cuda.get_device_name(0).replace(" ", "_")
    cache = tmp_path / "tune"
    cache.write_text("".join(f"{gpu}|dslash32q|{st}|0|{n}|{L}x{T} {variant}\n"
                             for L, T, _, _, rhs in SHAPES + SMALL for n in rhs for st in range(4)))
    r = subprocess.run([sys.executable, "-c", CHILD % {"root": ROOT, "shapes": SHAPES + SMALL}],
                       env=dict(os.environ, QS_TUNE_CACHE=str(cache)), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert len(cache.read_text().splitlines()) == 11 * 4   # nothing was timed: the forced one ran


CHILD64 = r"""
import sys
sys.path[:0] = [%(root)r, %(root)r + "/tests"]
import numpy as np
import torch
import paper_2108_11989_gb300 as qs
from oracle.dirac import WilsonDirac
from synth_inputs import make_config, random_spinor
for L, T, mask, anti, rhs in %(shapes)r:
    cfg = make_config(T=T, L=L, eps=0.6, theta_sigma=0.4, csw_su3=1.9, csw_u1=1.0, seed=3, cstar_mask=mask,
                      t_antiperiodic=anti)
    lat = qs.Lattice(L, T, mask, anti)
    lat.load_gauge(cfg.su3, cfg.theta, cfg.csw_su3, cfg.csw_u1)
    op, ns = WilsonDirac(cfg), cfg.n_sites
    for nrhs in rhs:
        psi = random_spinor(7, T, L, nrhs)
        ref = np.stack([op.apply_D(psi[r].reshape(-1), 0.07) for r in range(nrhs)]).reshape(nrhs, ns, 12)
        x = torch.from_numpy(np.ascontiguousarray(psi).view(np.float64).copy()).cuda().reshape(-1)
        for tiled in (False, True):
            xin = qs.to_tiled(x, ns) if tiled else x
            y = torch.full_like(xin, float("nan"))
            lat.apply_Dw(0.07, xin, y, tiled=tiled)
            y = qs.from_tiled(y, ns) if tiled else y
            got = y.cpu().numpy().view(np.complex128).reshape(nrhs, ns, 12)
            assert np.abs(got - ref).max() <= 1e-13 * np.abs(ref).max(), (L, T, nrhs, tiled)
    lat.close()
"""


@pytest.mark.parametrize("variant", range(3))
def test_forced_fp64_variant_matches_oracle(variant, tmp_path):
    import torch
    gpu = torch.cuda.get_device_name(0).replace(" ", "_")
    cache = tmp_path / "tune"
    cache.write_text("".join(f"{gpu}|dslash64s|{soa}|0|{n}|{L}x{T} {variant}\n"
                             for L, T, _, _, rhs in SHAPES + SMALL for n in rhs for soa in range(2)))
    r = subprocess.run([sys.executable, "-c", CHILD64 % {"root": ROOT, "shapes": SHAPES + SMALL}],
                       env=dict(os.environ, QS_TUNE_CACHE=str(cache)), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert len(cache.read_text().splitlines()) == 11 * 2
