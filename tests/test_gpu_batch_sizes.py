"""The batched operator in both its forms (a block per 32 sites for small batches, the persistent
one for large): the same bits as the operator on each lattice alone.

Lattices whose physical sites fill no tile of 32 or 128 (24, 1080, 3000), one to eight items with
uneven numbers of vectors and a mass per vector, and batches on both sides of the rule's line (32768
physical sites x vectors).
"""
import pytest

from synth_inputs import make_config

pytestmark = pytest.mark.gpu
BATCHES = [[(2, 3, 1)], [(2, 3, 5), (6, 5, 3), (4, 3, 16)], [(4, 4, 1), (2, 2, 1)] * 4, [(8, 8, 4), (8, 8, 4)],
           [(8, 8, 4), (8, 8, 4), (2, 3, 1)], [(10, 3, 11), (6, 5, 1)]]


@pytest.mark.parametrize("prec", ["f32", "canon", "f16", "bf16"])
@pytest.mark.parametrize("batch", BATCHES, ids=str)
def test_batch_equals_single_applications(batch, prec):
    import torch
    import paper_2108_11989_gb300 as qs
    p = {"f16": qs.QS_F16, "bf16": qs.QS_BF16}.get(prec, qs.QS_F32)
    g = torch.Generator(device="cuda")
    g.manual_seed(len(batch))
    lats, entries, want = {}, [], []
    for i, (L, T, n) in enumerate(batch):
        if (L, T) not in lats:
            cfg = make_config(T=T, L=L, eps=0.6, theta_sigma=0.4, csw_su3=1.9, csw_u1=1.0, seed=L + T, cstar_mask=0b011,
                              t_antiperiodic=True)
            lats[L, T] = qs.Lattice(L, T, 0b011, True)
            lats[L, T].load_gauge(cfg.su3, cfg.theta, cfg.csw_su3, cfg.csw_u1)
        lat = lats[L, T]
        x = torch.randn(n * lat.n_sites * 24, device="cuda", generator=g)
        if p != qs.QS_F32:
            q = torch.empty(n * lat.n_sites * qs.Q16_BYTES_PER_SITE, dtype=torch.uint8, device="cuda")
            qs.convert_spinors(lat.h, x, qs.QS_F32, q, p, n)
            x = q
        y, ref = torch.zeros_like(x), torch.zeros_like(x)
        masses = [0.1 * r - 0.3 - 0.01 * i for r in range(n)]
        step = x.numel() // n
        for r in range(n):
            lat.apply_Q(masses[r], x[r * step:(r + 1) * step], ref[r * step:(r + 1) * step], tiled=prec != "canon", prec=p)
        entries.append((lat, x, y, masses))
        want.append(ref)
    torch.cuda.synchronize()
    qs.apply_Q_batch(entries, tiled=prec != "canon", prec=p, stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    for (_, _, y, _), ref in zip(entries, want):
        assert torch.equal(y, ref)
    for lat in lats.values():
        lat.close()
