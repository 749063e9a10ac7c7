"""The work a user has this framework do, as cases that can be timed and compared.

A case is a dict of plain values.  `prepare` makes the inputs of one (gauge field, spinors,
lattice handle) from a seed, `run` does one pass through the public entry points, `exact`
gives the same outputs in 64 bits by plain torch, and `work` counts what the pass cannot do
without.  Gauge fields follow the synthetic ensembles of this repository: SU(3) links
exp(i eps H) with H Gaussian in the Lie algebra, U(1) angles N(0, 0.3^2), C* boundaries in
space, periodic time, c_sw = 1.9 (SU(3)) and 1.0 (U(1)), kappa around 0.135.
"""
import math

import numpy as np
import torch

import paper_2108_11989_gb300 as qs

PREC = {"f64": qs.QS_F64, "f32": qs.QS_F32, "f16": qs.QS_F16, "bf16": qs.QS_BF16}
CSW, CSW1, SIGMA1 = 1.9, 1.0, 0.3


def listed():
    return [
        # one application of Q to one vector on the smallest lattice: launch and call latency
        dict(name="q_tiny", kind="op", L=4, T=4, prec="f32", layout="canon", nrhs=1, gamma5=1, eps=0.3, kappa=0.135),
        # odd time extent, a row that is no multiple of a tile, bf16 storage, odd block of vectors
        dict(name="q_ragged", kind="op", L=10, T=7, prec="bf16", layout="tiled", nrhs=5, gamma5=1, eps=0.3, kappa=0.13),
        # the Chebyshev filter's operator: half of a block of 32 (C* pairing), 16-bit storage
        dict(name="q_filter", kind="op", L=16, T=32, prec="f16", layout="tiled", nrhs=16, gamma5=1, eps=0.2, kappa=0.135),
        # the inner CG's operator: half of a block of 32 in FP32
        dict(name="q_cg", kind="op", L=16, T=32, prec="f32", layout="tiled", nrhs=16, gamma5=1, eps=0.2, kappa=0.135),
        # the Rayleigh-Ritz operator: the whole block of 32 in FP64
        dict(name="q_rr", kind="op", L=16, T=32, prec="f64", layout="tiled", nrhs=32, gamma5=1, eps=0.2, kappa=0.135),
        # the largest lattice, filter storage, a block of 24
        dict(name="q_large", kind="op", L=32, T=64, prec="f16", layout="tiled", nrhs=24, gamma5=1, eps=0.15, kappa=0.135),
        # three configurations of uneven volume, many masses, one launch
        dict(name="q_batch", kind="batch", shapes="8x16,12x10,16x32", nrhs="8,5,16", prec="f32", layout="tiled",
             eps=0.2, kappa=0.135),
        # a quark propagator column pair: even-odd preconditioned solve in FP64
        dict(name="solve", kind="solve", L=12, T=24, nrhs=2, tol=1e-12, eps=0.2, kappa=0.135),
        # one stochastic estimate of the mass reweighting factor
        dict(name="w_mass", kind="w_mass", L=8, T=16, nsrc=2, n=3, tol=1e-12, eps=0.2, kappa=0.135),
        # low modes at one mass, cold start, converged far enough to be quoted
        dict(name="lowmodes", kind="lowmodes", L=12, T=24, k=16, nwant=4, tol=1e-8, degree=48, prec="f16", eps=0.2,
             kappa=0.135),
        # the headline: the sign of the Pfaffian of one configuration by the mass flow, followed until
        # the low modes have left the neighbourhood of zero
        dict(name="sign", kind="sign", L=8, T=12, k=32, nwant=2, tol=1e-5, degree=48, prec="f16", m0_max=0.5, eps=0.2,
             kappa=0.135),
        # training the step-proposal network: four Adam steps on minibatches; the losses and the
        # gradients at the weights that the steps before the last one left
        dict(name="mlp_train", kind="mlp", batch=512, n_hidden=128, steps=4),
    ]


def _even(rng, lo, hi):
    """An even number, its logarithm spread over [lo, hi]."""
    return 2 * max(1, round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2))


def _log(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo - 0.49), math.log(hi + 0.49))))))


def draw(rng):
    kind = rng.choice(["op", "op", "op", "op", "batch", "solve", "w_mass", "lowmodes", "sign", "mlp"])
    c = dict(kind=kind, eps=round(rng.uniform(0.15, 0.3), 3), kappa=round(rng.uniform(0.13, 0.135), 4))
    if kind == "op":
        c["prec"] = rng.choice(["f64", "f32", "f32", "f16", "bf16"])
        c["layout"] = rng.choice(["tiled", "canon"]) if c["prec"] in ("f64", "f32") else "tiled"
        c["gamma5"] = rng.choice([0, 1])
        top = 24 if c["prec"] == "f64" else 32
        c["L"], c["T"] = _even(rng, 4, top), _log(rng, 3, 2 * top)
        c["nrhs"] = _log(rng, 1, 32)
    elif kind == "batch":
        n = rng.randint(2, 8)
        c["prec"] = rng.choice(["f64", "f32", "f16", "bf16"])
        c["layout"] = rng.choice(["tiled", "canon"]) if c["prec"] in ("f64", "f32") else "tiled"
        c["shapes"] = ",".join("%dx%d" % (_even(rng, 4, 16), _log(rng, 3, 32)) for _ in range(n))
        c["nrhs"] = ",".join(str(_log(rng, 1, 16)) for _ in range(n))
    elif kind == "solve":
        c.update(L=_even(rng, 4, 12), T=_even(rng, 4, 24), nrhs=_log(rng, 1, 4), tol=1e-12)
    elif kind == "w_mass":
        c.update(L=_even(rng, 4, 8), T=_even(rng, 4, 16), nsrc=_log(rng, 1, 3), n=rng.randint(1, 3), tol=1e-12)
    elif kind == "lowmodes":
        c.update(L=_even(rng, 4, 12), T=_log(rng, 4, 24), k=rng.choice([12, 16]), nwant=rng.choice([2, 4]), tol=1e-8,
                 degree=rng.choice([24, 48]), prec=rng.choice(["f32", "f16", "bf16"]))
    elif kind == "sign":
        c.update(L=_even(rng, 4, 8), T=_log(rng, 4, 12), k=32, nwant=2, tol=1e-5, degree=48, m0_max=0.5,
                 prec=rng.choice(["f32", "f16", "bf16"]), eps=round(rng.uniform(0.18, 0.22), 3), kappa=0.135)
    else:
        c = dict(kind="mlp", batch=_log(rng, 16, 512), n_hidden=rng.choice([64, 96, 128]), steps=rng.randint(1, 4))
    return c


# ---- inputs --------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _mm(a, b):
    """3 x 3 complex products over the leading axes."""
    return sum(a[..., :, k, None] * b[..., None, k, :] for k in range(3))


def _gell_mann():
    m = np.zeros((8, 3, 3), dtype=np.complex128)
    m[0][0, 1] = m[0][1, 0] = m[3][0, 2] = m[3][2, 0] = m[5][1, 2] = m[5][2, 1] = 1
    m[1][0, 1] = m[4][0, 2] = m[6][1, 2] = -1j
    m[1][1, 0] = m[4][2, 0] = m[6][2, 1] = 1j
    m[2][0, 0], m[2][1, 1] = 1, -1
    m[7] = np.diag([1, 1, -2]) / np.sqrt(3)
    return torch.from_numpy(m).cuda()


def _field(L, T, eps, seed):
    """su3 [T,L,L,L,4,3,3] complex128 and theta [T,L,L,L,4] on the GPU."""
    g = _gen(seed)
    basis = _gell_mann().reshape(8, 9) / 2
    u = torch.empty((T, L, L, L, 4, 3, 3), dtype=torch.complex128, device="cuda")
    one = torch.eye(3, dtype=torch.complex128, device="cuda")
    for t in range(T):
        h = torch.randn((L, L, L, 4, 8), dtype=torch.float64, device="cuda", generator=g)
        x = 1j * eps * (h.to(torch.complex128) @ basis).reshape(L, L, L, 4, 3, 3)
        e = one + x / 20
        for n in range(19, 0, -1):   # exp by its series, |x| < 2
            e = one + _mm(x, e) / n
        u[t] = e
    th = SIGMA1 * torch.randn((T, L, L, L, 4), dtype=torch.float64, device="cuda", generator=g)
    return u, th


def _lattice(L, T, eps, seed, stream=None):
    u, th = _field(L, T, eps, seed)
    lat = qs.Lattice(L, T, stream=torch.cuda.current_stream() if stream is None else stream)
    lat.load_gauge(u.cpu().numpy(), th.cpu().numpy(), CSW, CSW1)
    return lat


def _m0(c):
    return 1.0 / (2.0 * c["kappa"]) - 4.0


def _tiled(x, nrhs, ns):
    """[nrhs][site][12][2] -> [nrhs][site / 16][12][site % 16][2]"""
    return x.reshape(nrhs, ns // 16, 16, 12, 2).transpose(2, 3).contiguous()


def _canon(x, nrhs, ns):
    return x.reshape(nrhs, ns // 16, 12, 16, 2).transpose(2, 3).reshape(nrhs, ns, 12, 2)


def _half(prec):
    return torch.float16 if prec == "f16" else torch.bfloat16


def _pack16(x, nrhs, ns, prec):
    """FP32 canonical spinors in the tiled 16-bit storage: per tile of 16 sites 12 x 16 pairs of
    16-bit reals, each divided by the site's largest component, then the 16 FP32 scales."""
    out = torch.empty((nrhs, ns // 16, 832), dtype=torch.uint8, device="cuda")
    for r in range(nrhs):
        v = x[r].reshape(ns // 16, 16, 12, 2)
        s = v.abs().amax(dim=(2, 3))
        q = (v * (1.0 / s)[:, :, None, None]).to(_half(prec)).transpose(1, 2).contiguous()
        out[r, :, :768] = q.reshape(ns // 16, 384).view(torch.uint8)
        out[r, :, 768:] = s.contiguous().view(torch.uint8).reshape(ns // 16, 64)
    return out


def _spinors(nrhs, ns, seed, dtype=torch.float32):
    """Canonical Gaussian spinors [nrhs][site][12][2] of unit variance per complex entry."""
    g = _gen(seed)
    x = torch.empty((nrhs, ns, 12, 2), dtype=dtype, device="cuda")
    for r in range(nrhs):
        x[r] = torch.randn((ns, 12, 2), dtype=dtype, device="cuda", generator=g) * 0.5 ** 0.5
    return x


def _stored(x, prec, layout, nrhs, ns):
    if prec in ("f16", "bf16"):
        return _pack16(x, nrhs, ns, prec)
    return _tiled(x, nrhs, ns) if layout == "tiled" else x.contiguous()


def _outputs(y, prec):
    """The output buffer, or its mantissas and scales in 16-bit storage (views)."""
    if prec in ("f16", "bf16"):
        return [y[..., :768].view(_half(prec)), y[..., 768:].view(torch.float32)]
    return y


def _op_state(L, T, nrhs, c, seed):
    lat = _lattice(L, T, c["eps"], seed)
    ns = lat.n_sites
    x = _spinors(nrhs, ns, seed + 1, torch.float64 if c["prec"] == "f64" else torch.float32)
    x = _stored(x, c["prec"], c["layout"], nrhs, ns)
    y = torch.empty_like(x)
    return lat, x, y, _outputs(y, c["prec"])


def _batch(c):
    return [(tuple(int(v) for v in s.split("x")), int(n)) for s, n in zip(c["shapes"].split(","), c["nrhs"].split(","))]


def _masses(c, i, n):
    return [_m0(c) + 0.01 * ((7 * r + 3 * i) % 5) for r in range(n)]


def _shifts(n):
    """Shifts of a rational approximation on |Q_hat| in [0.02, 8]: a staircase in the logarithm."""
    s = np.exp(np.linspace(math.log(0.05), math.log(4.0), 2 * n))
    return s[1::2].copy(), s[0::2].copy()   # nu, mu


def _mlp_data(c, seed):
    r = np.random.default_rng(seed)
    ni, nh, no = 192, c["n_hidden"], 25
    p = [r.standard_normal((nh, ni)) / ni ** 0.5, 0.05 * r.standard_normal(nh), r.standard_normal((nh, nh)) / nh ** 0.5,
         0.05 * r.standard_normal(nh), r.standard_normal((no, nh)) / nh ** 0.5, 0.05 * r.standard_normal(no)]
    x = r.standard_normal((c["steps"], c["batch"], ni)).astype(np.float32)
    t = np.concatenate([r.standard_normal((c["steps"], c["batch"], 1)), r.random((c["steps"], c["batch"], no - 1)) < 0.3], 2)
    return [a.astype(np.float32) for a in p], x, t.astype(np.float32)


def prepare(case, seed):
    c, kind = case, case["kind"]
    seed = 7919 * int(seed) + 13
    if kind == "op":
        lat, x, y, out = _op_state(c["L"], c["T"], c["nrhs"], c, seed)
        return dict(kind=kind, lat=lat, m0=_m0(c), x=x, y=y, out=out, tiled=c["layout"] == "tiled", prec=PREC[c["prec"]],
                    apply=lat.apply_Q if c["gamma5"] else lat.apply_Dw)
    if kind == "batch":
        entries, out = [], []
        for i, ((L, T), n) in enumerate(_batch(c)):
            lat, x, y, o = _op_state(L, T, n, c, seed + 100 * i)
            entries.append((lat, x, y, _masses(c, i, n)))
            out.append(o)
        return dict(kind=kind, entries=entries, out=out, tiled=c["layout"] == "tiled", prec=PREC[c["prec"]],
                    stream=torch.cuda.current_stream())
    if kind == "mlp":
        p, x, t = _mlp_data(c, seed)
        net = qs.MLP(192, c["n_hidden"], 25, max_batch=c["batch"], stream=torch.cuda.current_stream())
        return dict(kind=kind, net=net, p=p, x=torch.from_numpy(x).cuda(), t=torch.from_numpy(t).cuda())
    if kind in ("solve", "w_mass"):
        lat = _lattice(c["L"], c["T"], c["eps"], seed)
        b = _spinors(c["nrhs"] if kind == "solve" else c["nsrc"], lat.n_sites, seed + 1, torch.float64)
        s = dict(kind=kind, lat=lat, m0=_m0(c), b=b, tol=c["tol"])
        if kind == "solve":
            s["x"] = torch.empty_like(b)
        else:
            s["nu"], s["mu"] = _shifts(c["n"])
        return s
    # eigensolver and flow run on a stream of their own (as a driver that overlaps
    # configurations does), where the filter can be replayed as a graph
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    lat = _lattice(c["L"], c["T"], c["eps"], seed, stream)
    eig = dict(k=c["k"], nwant=c["nwant"], tol=c["tol"], cheb_degree=c["degree"], precision=PREC[c["prec"]], max_iter=400,
               warm_start=0)
    opts = qs.eig_default_opts(**eig) if kind == "lowmodes" else qs.sign_default_opts(eig=eig, m0_max=c["m0_max"])
    torch.cuda.synchronize()
    return dict(kind=kind, lat=lat, stream=stream, m0=_m0(c), opts=opts, nwant=c["nwant"])


def run(state):
    s, kind = state, state["kind"]
    if kind == "op":
        s["apply"](s["m0"], s["x"], s["y"], tiled=s["tiled"], prec=s["prec"])
        return s["out"]
    if kind == "batch":
        qs.apply_Q_batch(s["entries"], tiled=s["tiled"], stream=s["stream"], prec=s["prec"])
        return s["out"]
    if kind == "solve":
        s["lat"].solve_D(s["m0"], s["b"], s["x"], tol=s["tol"])
        return s["x"]
    if kind == "w_mass":
        q, lw, _ = s["lat"].w_mass(s["m0"], s["m0"] + 0.002, s["nu"], s["mu"], s["b"], tol=s["tol"])
        return [q, np.array([lw])]
    if kind == "lowmodes":
        # the converged values (the others of the block are by-products without a tolerance)
        ev, _, _ = s["lat"].lowmodes_at_mass(s["m0"], s["opts"])
        return np.sort(np.abs(ev[:s["nwant"]]))
    if kind == "sign":
        sign, rep = s["lat"].pfaffian_sign(s["m0"], s["opts"])
        # lambda_bar at the target and after the first step (every flow has both); the
        # eigensolver's relative accuracy is 1e-5, so FP32 holds them
        return [sign, rep["crossings"], np.array(rep["lambda_bar"][:2], dtype=np.float32)]
    net = s["net"]
    net.set_params(s["p"])
    losses = [net.train_step(s["x"][i], s["t"][i], 2e-3) for i in range(len(s["x"]))]
    return [np.array(losses, dtype=np.float32)] + net.get_grads()


# ---- what a pass cannot do without -----------------------------------------------------------

_SPINOR = {"f64": 192, "f32": 96, "f16": 52, "bf16": 52}
_OP_FLOPS = 1872   # per doubled site: 1320 hopping, 504 SW term, 48 mass


def _op_work(L, T, nrhs, prec):
    ns = 2 * L ** 3 * T
    return ns * (2 * _SPINOR[prec] * nrhs + 72 * (8 if prec == "f64" else 4)), ns * nrhs * _OP_FLOPS


def work(case):
    c, kind = case, case["kind"]
    if kind == "op":
        b, f = _op_work(c["L"], c["T"], c["nrhs"], c["prec"])
    elif kind == "batch":
        w = [_op_work(L, T, n, c["prec"]) for (L, T), n in _batch(c)]
        b, f = sum(v[0] for v in w), sum(v[1] for v in w)
    elif kind == "mlp":
        n = 192 * c["n_hidden"] + c["n_hidden"] ** 2 + 25 * c["n_hidden"]
        b = c["steps"] * (c["batch"] * 217 * 4 + 7 * 4 * n)
        f = c["steps"] * (6 * c["batch"] * n - 2 * c["batch"] * 192 * c["n_hidden"])
    elif kind in ("solve", "w_mass"):
        # about 185 CG iterations on Q_hat^2 to 1e-12, each two D_hat (one operator each); two solves a factor
        it = 185 * (1 if kind == "solve" else 2 * c["n"])
        n = c["nrhs"] if kind == "solve" else c["nsrc"]
        ns = 2 * c["L"] ** 3 * c["T"]
        b = it * ns * (576 + 5 * 96 * n)   # fields once, five half-lattice vectors read or written
        f = it * ns * n * 2 * _OP_FLOPS
    else:
        # operator applications of one eigensolve: about six filters of degree d over the block
        ns = 2 * c["L"] ** 3 * c["T"]
        solves = 1 if kind == "lowmodes" else 6
        n = solves * 6 * 2 * c["degree"] * c["k"] // 2
        b, f = n * ns * (2 * 52 + 288 * 2 // c["k"]), n * ns * _OP_FLOPS
    return {"bytes": float(b), "flops": float(f)}


# ---- the same in 64 bits, by plain torch --------------------------------------------------------


def _gammas():
    s = torch.tensor([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=torch.complex128, device="cuda")
    z, e = torch.zeros(2, 2, dtype=torch.complex128, device="cuda"), torch.eye(2, dtype=torch.complex128, device="cuda")
    block = lambda a, b: torch.cat([torch.cat([z, a], 1), torch.cat([b, z], 1)], 0)  # noqa: E731
    return [block(-e, -e)] + [block(-1j * s[k], 1j * s[k]) for k in range(3)]


def _shift(f, mu, step, L):
    """f at x + step mu on the doubled lattice [T, L(z), L(y), 2L(x), ...] with C* in y and z."""
    if mu == 0:
        return torch.roll(f, -step, 0)
    if mu == 1:
        return torch.roll(f, -step, 3)
    dim = 2 if mu == 2 else 1
    g = torch.roll(f, -step, dim)
    edge = f.shape[dim] - 1 if step > 0 else 0
    w = g.narrow(dim, edge, 1)
    w.copy_(torch.roll(w, L, 3))
    return g


class _Dirac:
    """D(m0) on the doubled lattice in 64 bits, spinors [T, L, L, 2L, 4, 3]."""

    def __init__(self, L, T, eps, seed):
        u, th = _field(L, T, eps, seed)
        self.L, self.gam = L, _gammas()
        u = torch.cat([u, u.conj()], 3)
        th = torch.cat([th, -th], 3)
        ph = torch.exp(1j * th)
        self.A = self._clover(u, ph)
        self.V = u * ph[..., None, None]
        e = torch.eye(4, dtype=torch.complex128, device="cuda")
        self.Pm, self.Pp = [e - g for g in self.gam], [e + g for g in self.gam]

    def _leaves(self, u, mu, nu, mul, dag):
        L = self.L
        um, un = u(mu), u(nu)
        sh = lambda f, m, s: _shift(f, m, s, L)  # noqa: E731
        um_pn, un_pm = sh(um, nu, 1), sh(un, mu, 1)
        plaq = mul(mul(um, un_pm), mul(dag(um_pn), dag(un)))
        um_mm, un_mm = sh(um, mu, -1), sh(un, mu, -1)
        l2 = mul(mul(un, dag(sh(um_pn, mu, -1))), mul(dag(un_mm), um_mm))
        um_mn, un_mn = sh(um, nu, -1), sh(un, nu, -1)
        l3 = mul(mul(dag(um_mm), dag(sh(un_mm, nu, -1))), mul(sh(um_mm, nu, -1), un_mn))
        l4 = mul(mul(dag(un_mn), um_mn), mul(sh(un_pm, nu, -1), dag(um)))
        return plaq + l2 + l3 + l4

    def _clover(self, u, ph):
        """The two 6 x 6 chiral blocks of A = (i / 2) sum_{mu < nu} sigma_{mu nu} F_{mu nu}."""
        A = torch.zeros(u.shape[:4] + (2, 2, 3, 2, 3), dtype=torch.complex128, device="cuda")
        eye = torch.eye(3, dtype=torch.complex128, device="cuda")
        dag = lambda m: m.conj().transpose(-1, -2)  # noqa: E731
        for mu in range(4):
            for nu in range(mu + 1, 4):
                q = self._leaves(lambda d: u[..., d, :, :], mu, nu, _mm, dag)
                F = CSW / 8 * (q - dag(q))
                q1 = self._leaves(lambda d: ph[..., d], mu, nu, lambda a, b: a * b, torch.conj)
                F = F + CSW1 / 8 * (q1 - q1.conj())[..., None, None] * eye
                sig = 0.5j * (self.gam[mu] @ self.gam[nu] - self.gam[nu] @ self.gam[mu])
                for b in range(2):
                    for i in range(2):
                        for j in range(2):
                            s = complex(sig[2 * b + i, 2 * b + j])
                            if s != 0:
                                A[..., b, i, :, j, :] += 0.5j * s * F
        return A.reshape(u.shape[:4] + (2, 6, 6))

    def hop(self, p):
        out = torch.zeros_like(p)
        for mu in range(4):
            v = self.V[..., mu, :, :]
            f = torch.einsum("ab,tzyxbc->tzyxac", self.Pm[mu], _shift(p, mu, 1, self.L))
            out += sum(f[..., :, k, None] * v[..., None, :, k] for k in range(3))
            f = torch.einsum("ab,tzyxbc->tzyxac", self.Pp[mu], p)
            f = sum(f[..., :, k, None] * v[..., None, k, :].conj() for k in range(3))
            out += _shift(f, mu, -1, self.L)
        return -0.5 * out

    def site(self, p, m0, A=None):
        q = p.reshape(p.shape[:4] + (2, 6))
        q = (4 + m0) * q + torch.einsum("tzyxbij,tzyxbj->tzyxbi", self.A, q) if A is None else \
            torch.einsum("tzyxbij,tzyxbj->tzyxbi", A, q)
        return q.reshape(p.shape)

    def D(self, p, m0):
        return self.site(p, m0) + self.hop(p)


def _g5(p):
    p = p.clone()
    p[..., 2:, :] *= -1
    return p


def _cg(A, b, tol=1e-14, cap=3000):
    x, r = torch.zeros_like(b), b.clone()
    p, rr = r.clone(), float((b.conj() * b).real.sum())
    stop = tol * tol * rr
    for _ in range(cap):
        if rr <= stop:
            break
        q = A(p)
        a = rr / float((p.conj() * q).real.sum())
        x += a * p
        r -= a * q
        n = float((r.conj() * r).real.sum())
        p = r + (n / rr) * p
        rr = n
    return x


def _decode(x, prec, layout, nrhs, ns):
    """Stored spinors as FP64 canonical ones."""
    if prec in ("f16", "bf16"):
        s = x[..., 768:].contiguous().view(torch.float32).reshape(nrhs, ns // 16, 1, 16, 1).double()
        v = x[..., :768].contiguous().view(_half(prec)).reshape(nrhs, ns // 16, 12, 16, 2).double()
        return _canon(v * s, nrhs, ns)
    return (_canon(x, nrhs, ns) if layout == "tiled" else x).double()


def _exact_op(c, L, T, nrhs, masses, gamma5, seed):
    d, ns = _Dirac(L, T, c["eps"], seed), 2 * L ** 3 * T
    x = _spinors(nrhs, ns, seed + 1, torch.float64 if c["prec"] == "f64" else torch.float32)
    out, scales, half = [], [], c["prec"] in ("f16", "bf16")
    for r in range(nrhs):
        one = _decode(_stored(x[r:r + 1], c["prec"], c["layout"], 1, ns), c["prec"], c["layout"], 1, ns)
        y = d.D(torch.view_as_complex(one.contiguous()).reshape(T, L, L, 2 * L, 4, 3), masses[r])
        y = torch.view_as_real(_g5(y) if gamma5 else y).reshape(1, ns, 12, 2)
        y = _tiled(y, 1, ns) if c["layout"] == "tiled" else y
        if half:
            s = y.abs().amax(dim=(2, 4))
            y = (y / s[:, :, None, :, None]).reshape(1, ns // 16, 384)
            scales.append(s)
        out.append(y)
    return [torch.cat(out), torch.cat(scales)] if half else torch.cat(out)


def _exact_solve(c, seed):
    L, T = c["L"], c["T"]
    d, ns, m0 = _Dirac(L, T, c["eps"], seed), 2 * L ** 3 * T, _m0(c)
    b = torch.view_as_complex(_spinors(c["nrhs"], ns, seed + 1, torch.float64)).reshape(c["nrhs"], T, L, L, 2 * L, 4, 3)
    Q = lambda p: _g5(d.D(p, m0))  # noqa: E731
    x = torch.stack([Q(_cg(lambda p: Q(Q(p)), _g5(b[r]))) for r in range(c["nrhs"])])
    return torch.view_as_real(x).reshape(c["nrhs"], ns, 12, 2)


def _exact_w_mass(c, seed):
    L, T, m = c["L"], c["T"], _m0(c)
    d, ns, mp = _Dirac(L, T, c["eps"], seed), 2 * L ** 3 * T, _m0(c) + 0.002
    ar = [torch.arange(n, device="cuda") for n in (T, L, L, 2 * L)]
    odd = (ar[0][:, None, None, None] + ar[1][:, None, None] + ar[2][:, None] + ar[3]) % 2 == 1
    even = (~odd)[..., None, None].double()
    odd = odd[..., None, None].double()
    eye = torch.eye(6, dtype=torch.complex128, device="cuda")
    inv = {q: torch.linalg.inv(d.A + (4 + q) * eye) for q in (m, mp)}

    def dhat(p, q):
        u = d.site(odd * d.hop(p), q, inv[q])
        return even * (d.site(p, q) - d.hop(u))

    def shifted(p, q, s):
        Q = lambda v: _g5(dhat(v, q))  # noqa: E731
        y = _cg(lambda v: Q(Q(v)) + s * s * v, _g5(p))
        return Q(y) - 1j * s * y

    nu, mu = _shifts(c["n"])
    q = np.zeros((c["n"], c["nsrc"]))
    eta = torch.view_as_complex(_spinors(c["nsrc"], ns, seed + 1, torch.float64)).reshape(c["nsrc"], T, L, L, 2 * L, 4, 3)
    for l in range(c["nsrc"]):
        e = even * eta[l]
        for j in range(c["n"]):
            v = 1j * (mu[j] - nu[j]) * _g5(shifted(e, m, nu[j]))
            v = shifted(v, mp, mu[j])
            x = dhat(v, mp) - dhat(v, m)
            q[j, l] = 2 * float((e.conj() * x).real.sum()) + float((x.conj() * x).real.sum())
    top = (-q).max(axis=1, keepdims=True)
    return [q, np.array([float((top[:, 0] + np.log(np.exp(-q - top).mean(axis=1))).sum())])]


def _exact_mlp(c, seed):
    p, x, t = _mlp_data(c, seed)
    p = [torch.from_numpy(a).cuda().double().requires_grad_(True) for a in p]
    x, t = torch.from_numpy(x).cuda().double(), torch.from_numpy(t).cuda().double()
    m, v, losses = [torch.zeros_like(a) for a in p], [torch.zeros_like(a) for a in p], []
    for i in range(c["steps"]):
        h = torch.relu(x[i] @ p[0].T + p[1])
        y = torch.relu(h @ p[2].T + p[3]) @ p[4].T + p[5]
        sp = torch.nn.functional.softplus(y[:, 1:], threshold=100)
        loss = (0.5 * (y[:, 0] - t[i, :, 0]) ** 2 + (sp - t[i, :, 1:] * y[:, 1:]).sum(1)).mean()
        grad = torch.autograd.grad(loss, p)
        losses.append(float(loss))
        with torch.no_grad():
            for a, g, b, w in zip(p, grad, m, v):
                b.mul_(0.9).add_(0.1 * g)
                w.mul_(0.999).add_(0.001 * g * g)
                a -= 2e-3 * (b / (1 - 0.9 ** (i + 1))) / (torch.sqrt(w / (1 - 0.999 ** (i + 1))) + 1e-8)
    return [np.array(losses)] + [g.cpu().numpy() for g in grad]


def exact(case, seed):
    c, kind = case, case["kind"]
    seed = 7919 * int(seed) + 13
    if kind == "op":
        return _exact_op(c, c["L"], c["T"], c["nrhs"], [_m0(c)] * c["nrhs"], c["gamma5"], seed)
    if kind == "batch":
        return [_exact_op(c, L, T, n, _masses(c, i, n), 1, seed + 100 * i) for i, ((L, T), n) in enumerate(_batch(c))]
    if kind == "solve":
        return _exact_solve(c, seed)
    if kind == "w_mass":
        return _exact_w_mass(c, seed)
    if kind == "mlp":
        return _exact_mlp(c, seed)
    return None   # eigenvalues of matrices far too large for a dense solve
