"""The launch variants of the plain operator and of the operator with the CG's sums are chosen apart:
a CG that times the latter leaves the choice of the former open."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
sys.path[:0] = [%(root)r, %(root)r + "/tests"]
import ctypes
import torch
import internals
import paper_2108_11989_gb300 as qs
from synth_inputs import make_config
lib = internals.load()
cfg = make_config(T=4, L=4, eps=0.5, theta_sigma=0.3, csw_su3=1.5, csw_u1=1.0, seed=2)
lat = qs.Lattice(4, 4)
lat.load_gauge(cfg.su3, cfg.theta, cfg.csw_su3, cfg.csw_u1)
b = torch.randn((3, cfg.n_sites * 24), device="cuda")
x, n = torch.empty_like(b), (ctypes.c_int64 * 3)()
torch.cuda.synchronize()
assert lib.t_cg(lat.h, 3, 0.1, 1e-3, 100, b.data_ptr(), x.data_ptr(), n) == 0
"""


def test_sums_do_not_take_the_plain_slot(tmp_path):
    cache = tmp_path / "tune"
    r = subprocess.run([sys.executable, "-c", CHILD % {"root": ROOT}], env=dict(os.environ, QS_TUNE_CACHE=str(cache)),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    forms = [line.split("|")[2:5] for line in cache.read_text().splitlines()]
    assert forms == [["0", "2", "3"]], forms   # tiled FP32, with sums, three vectors; nothing else timed
