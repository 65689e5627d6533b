"""The work that a user of this library has it do, as cases that can be timed.

Every case goes through the public binding (`paper_1702_00124_gb300.wdhmc` and
`.autograd`).  Kinds:

  khat        mdagm_apply: K_hat on one or more half spinors
  cg          cg_solve of K_hat, or of K_hat P(K_hat) when poly_n > 0
  force       fermion_force of one pseudofermion term (its solve included)
  autograd    the action and its force through torch.autograd
  gauge_md    links in, gauge-only molecular dynamics, links out
  batch_cg    many lattices x right-hand sides in one batched CG
  trajectory  links in, one HMC trajectory of the PF-MP action, links out

Sizes are the library's workloads (4^4, 8^3 x 16, 16^3 x 32, 32^3 x 64, the 24
uneven lattices) and ragged ones of the same range.  Links are exp(i a H) with H
a Gaussian traceless Hermitian matrix, spinors and momenta Gaussian.

The library returns FP64 storage whatever arithmetic was asked for.  Where a
case asks for FP32 arithmetic, `run` hands the result on as float32, the
type that the values have; solutions (true residual 1e-10) stay float64.
"""
import math

import torch

from paper_1702_00124_gb300 import wdhmc as wd
from paper_1702_00124_gb300.autograd import pf_action

PREC = {"f64": wd.F64, "f32": wd.F32, "f16": wd.F16, "bf16": wd.BF16}
KIND = {"plain": wd.PLAIN, "hasenbusch": wd.HASENBUSCH, "poly": wd.POLY, "filtered": wd.FILTERED}
EPS, LAM = 0.005, 8.0          # interval of the Chebyshev filter in every workload
LAM_2MN = 0.1931833275037836   # Omelyan 2MN
# iterations of a solve to 1e-10 that `work` counts (kappa and the links decide the true number)
ITERS, ITERS_FILTERED = 60, 20


def _dims(c):
    return tuple(c[k] for k in ("lx", "ly", "lz", "lt"))


def _case(kind, dims, **kw):
    lx, ly, lz, lt = dims
    return dict(kind=kind, lx=lx, ly=ly, lz=lz, lt=lt, **kw)


def listed():
    return [
        # the smallest lattice, plain FP64: nothing but launches and latency
        dict(name="cg_f64_4x4x4x4", **_case("cg", (4, 4, 4, 4), prec="f64", recon=0, resid=0, kappa=0.12, a=0.3, poly_n=0)),
        # mixed precision on a small lattice, FP64 residuals: what a quick study runs
        dict(name="cg_f32_8x8x8x16", **_case("cg", (8, 8, 8, 16), prec="f32", recon=1, resid=0, kappa=0.13, a=0.5, poly_n=0)),
        # 16-bit spinors on a lattice whose rows do not fill a warp
        dict(name="cg_bf16_12x12x12x24", **_case("cg", (12, 12, 12, 24), prec="bf16", recon=1, resid=1, kappa=0.13, a=0.4, poly_n=0)),
        # the plain method at the paper's volume: every operation in FP64
        dict(name="cg_f64_16x16x16x32", **_case("cg", (16, 16, 16, 32), prec="f64", recon=0, resid=0, kappa=0.135, a=0.5, poly_n=0)),
        # the stencil itself on the large lattice
        dict(name="khat_f32_32x32x32x64", **_case("khat", (32, 32, 32, 64), prec="f32", recon=1, nrhs=1, kappa=0.136, a=0.5)),
        # a ragged lattice with the default 18-real links and several right-hand sides
        dict(name="khat_f32_10x14x18x22_x3", **_case("khat", (10, 14, 18, 22), prec="f32", recon=0, nrhs=3, kappa=0.13, a=0.5)),
        # the filtered solve that most of a production trajectory consists of
        dict(name="filtered_cg_f32_32x32x32x64", **_case("cg", (32, 32, 32, 64), prec="f32", recon=1, resid=1, kappa=0.128, a=0.5, poly_n=24)),
        # the differentiated Hasenbusch action at the paper's volume, forward and backward
        dict(name="autograd_16x16x16x32", **_case("autograd", (16, 16, 16, 32), term="hasenbusch", prec="f32", recon=1, resid=1, kappa=0.135, kappa_h=0.125, a=0.5, poly_n=0)),
        # the polynomial term's force: no solve, K_hat and outer products
        dict(name="force_poly_16x16x16x32", **_case("force", (16, 16, 16, 32), term="poly", prec="f32", recon=1, resid=1, kappa=0.125, kappa_h=0.0, a=0.5, poly_n=16)),
        # link updates and gauge forces of a large lattice (thermalising a gauge field)
        dict(name="gauge_md_32x32x32x64", **_case("gauge_md", (32, 32, 32, 64), prec="f32", beta=5.6, steps=2, tau=0.1, a=0.5)),
        # 96 systems on 24 uneven lattices
        dict(name="batch_cg_24x4", kind="batch_cg", n_small=8, n_mid=8, n_large=8, nrhs=4, mode=1, a=0.4),
        # a whole PF-MP trajectory at the paper's volume
        dict(name="trajectory_16x16x16x32", **_case("trajectory", (16, 16, 16, 32), prec="f32", recon=1, resid=1, kappa=0.136, kappa_h=0.128, poly_n=24, beta=5.6, steps=4, tau=0.4, a=0.5)),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_dims(rng, vmin, vmax):
    """Even extents, volume spread over the logarithm of [vmin, vmax], aspect ratios up to about 2.5."""
    v = _log_uniform(rng, vmin, vmax)
    while True:
        e = [math.exp(rng.uniform(-0.45, 0.45)) for _ in range(4)]
        s = (v / math.prod(e)) ** 0.25
        d = [min(64, max(4, 2 * round(s * x / 2))) for x in e]
        if vmin <= math.prod(d) <= vmax:
            return tuple(d)


def draw(rng):
    kind = rng.choice(["khat", "khat", "cg", "cg", "filtered", "force", "autograd", "gauge_md", "batch_cg", "trajectory"])
    a = round(rng.uniform(0.3, 0.5), 3)
    kappa = round(rng.uniform(0.12, 0.136), 4)
    kappa_h = round(kappa - rng.uniform(0.005, 0.01), 4)
    prec = rng.choice(["f32", "f32", "f64"])
    recon, resid = rng.choice([0, 1, 1]), rng.choice([0, 1, 1])
    if kind == "khat":
        nrhs = rng.choice([1, 1, 2, 3, 4])
        return _case("khat", _draw_dims(rng, 256, 2097152 if nrhs == 1 else 500000), prec=prec, recon=recon, nrhs=nrhs, kappa=kappa, a=a)
    if kind == "cg":
        prec = rng.choice(["f64", "f32", "f32", "f16", "bf16"])
        return _case("cg", _draw_dims(rng, 256, 131072 if prec == "f64" else 1000000), prec=prec, recon=recon, resid=resid, kappa=kappa, a=a, poly_n=0)
    if kind == "filtered":
        return _case("cg", _draw_dims(rng, 4096, 1000000), prec="f32", recon=recon, resid=1, kappa=kappa, a=a, poly_n=rng.choice([8, 16, 24]))
    if kind == "force":
        term = rng.choice(["plain", "hasenbusch", "poly", "poly", "filtered"])
        return _case("force", _draw_dims(rng, 256, 20000 if prec == "f64" else 140000), term=term, prec=prec, recon=recon, resid=resid, kappa=kappa,
                     kappa_h=kappa_h, a=a, poly_n=rng.choice([8, 16, 24]))
    if kind == "autograd":
        return _case("autograd", _draw_dims(rng, 256, 140000), term=rng.choice(["plain", "hasenbusch"]), prec="f32", recon=recon, resid=resid,
                     kappa=kappa, kappa_h=kappa_h, a=a, poly_n=0)
    if kind == "gauge_md":
        return _case("gauge_md", _draw_dims(rng, 256, 1500000), prec=prec, beta=5.6, steps=rng.choice([1, 2, 3]), tau=0.1, a=a)
    if kind == "batch_cg":
        return dict(kind="batch_cg", n_small=rng.randint(1, 8), n_mid=rng.randint(0, 6), n_large=rng.randint(0, 5), nrhs=rng.choice([1, 2, 3, 4, 8]),
                    mode=rng.choice([1, 1, 0]), a=a)
    return _case("trajectory", _draw_dims(rng, 1024, 30000), prec="f32", recon=1, resid=1, kappa=kappa, kappa_h=kappa_h, poly_n=rng.choice([8, 16]), beta=5.6,
                 steps=rng.choice([1, 2]), tau=0.2, a=a)


# ---------------------------------------------------------------------------
# inputs

def _mm(A, B):
    return (A.unsqueeze(-1) * B.unsqueeze(-3)).sum(-2)


_T = torch.zeros(8, 3, 3, dtype=torch.complex128)      # generators lambda_a / 2
_T[0, 0, 1] = _T[0, 1, 0] = 0.5
_T[1, 0, 1], _T[1, 1, 0] = -0.5j, 0.5j
_T[2, 0, 0], _T[2, 1, 1] = 0.5, -0.5
_T[3, 0, 2] = _T[3, 2, 0] = 0.5
_T[4, 0, 2], _T[4, 2, 0] = -0.5j, 0.5j
_T[5, 1, 2] = _T[5, 2, 1] = 0.5
_T[6, 1, 2], _T[6, 2, 1] = -0.5j, 0.5j
_T[7, 0, 0] = _T[7, 1, 1] = 0.5 / math.sqrt(3)
_T[7, 2, 2] = -1.0 / math.sqrt(3)


def _alg(h):
    """[n, 8] coordinates -> [n, 3, 3] Hermitian traceless matrices."""
    return (h.to(torch.complex128) @ _T.to(h.device).reshape(8, 9)).reshape(-1, 3, 3)


def _expi(Q):
    """exp(i Q): Taylor series of the eighth of Q, squared three times."""
    A = (0.125j) * Q
    one = torch.eye(3, dtype=Q.dtype, device=Q.device)
    E = one + A / 14.0
    for k in range(13, 0, -1):
        E = one + _mm(A, E) / k
    for _ in range(3):
        E = _mm(E, E)
    return E


def _gen(seed, k):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + k)


def _randn(n, g):
    return torch.randn(n, dtype=torch.float64, device="cuda", generator=g)


def _links(dims, a, seed, k=0):
    """Lexicographic links [V * 36 complex] exp(i a H) as flat float64."""
    n = 4 * math.prod(dims)
    g = _gen(seed, k)
    out = torch.empty(n, 9, dtype=torch.complex128, device="cuda")
    for s in range(0, n, 1 << 20):
        m = min(n, s + (1 << 20))
        out[s:m] = _expi(a * _alg(_randn((m - s, 8), g))).reshape(-1, 9)
    return torch.view_as_real(out).reshape(-1)


def _lattice(c, U):
    lat = wd.Lattice(_dims(c))
    lat.wd_set_recon(c.get("recon", 0))
    lat.wd_gauge_load(U)
    if c.get("resid"):
        lat.wd_set_residual(1)
    return lat


def _params(c):
    return wd.cg_params(tol=1e-10, prec=PREC[c["prec"]], maxiter=20000)


def _term(c, name):
    poly = (c["poly_n"], EPS, LAM)
    if name == "hasenbusch":
        return wd.term(wd.HASENBUSCH, c["kappa"], c["kappa_h"])
    if name == "plain":
        return wd.term(wd.PLAIN, c["kappa"])
    return wd.term(KIND[name], c["kappa"], poly=poly)


BATCH_DIMS = ((8, 8, 8, 8), (12, 12, 12, 24), (16, 16, 16, 32))


def _batch_groups(c):
    return [(d, n) for d, n in zip(BATCH_DIMS, (c["n_small"], c["n_mid"], c["n_large"])) if n > 0]


def _batch_kappas(c, seed):
    n = sum(k for _, k in _batch_groups(c))
    g = torch.Generator().manual_seed(1000003 * int(seed) + 7)
    return (0.125 + 0.01 * torch.rand(n, dtype=torch.float64, generator=g)).tolist()


def _batch_inputs(c, seed):
    out, i = [], 0
    for d, n in _batch_groups(c):
        for _ in range(n):
            out.append((d, _links(d, c["a"], seed, 20 + 2 * i), _randn(c["nrhs"] * 12 * math.prod(d), _gen(seed, 21 + 2 * i))))
            i += 1
    return out


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    s = {"case": c}
    if kind == "batch_cg":
        ins = _batch_inputs(c, seed)
        lats = []
        for d, U, _ in ins:
            lats.append(_lattice(dict(lx=d[0], ly=d[1], lz=d[2], lt=d[3], recon=1, resid=1), U))
        s["lats"] = lats
        s["b"] = [b for _, _, b in ins]
        s["x"] = [torch.zeros_like(b) for b in s["b"]]
        s["batch"] = wd.Batch(lats, _batch_kappas(c, seed), [c["nrhs"]] * len(lats))
        s["params"] = wd.cg_params(tol=1e-10, prec=wd.F32)
        return s
    dims = _dims(c)
    U = _links(dims, c["a"], seed)
    s["lat"] = lat = _lattice(c, U)
    half = 12 * math.prod(dims)                      # reals of a half spinor
    g = _gen(seed, 1)
    if kind == "khat":
        s["in"] = _randn(c["nrhs"] * half, g)
        s["out"] = torch.empty_like(s["in"])
    elif kind == "cg":
        s["b"] = _randn(half, g)
        s["x"] = torch.zeros_like(s["b"])
        s["params"] = _params(c)
    elif kind in ("force", "autograd"):
        s["phi"] = _randn(half, g)
        s["params"], s["term"] = _params(c), _term(c, c["term"])
        if kind == "force":
            s["F"] = lat.algebra_field()
        else:
            s["w"] = torch.zeros(64 * lat.Vh, dtype=torch.float64, device="cuda", requires_grad=True)
    elif kind == "gauge_md":
        s["U"], s["Uout"] = U, torch.empty_like(U)
        s["P0"] = _randn(64 * lat.Vh, g)
        s["P"] = torch.empty_like(s["P0"])
        s["ops"] = wd.wd_schedule_nested(1, c["tau"], [-1], [c["steps"]])
        s["params"] = _params(c)
    else:
        s["U"], s["Uout"] = U, torch.empty_like(U)
        # outer group 0: filtered + Hasenbusch terms; group 1: polynomial term; -1: gauge action
        s["ops"] = wd.wd_schedule_nested(1, c["tau"], [0, 1, -1], [c["steps"], 1, 2])
        poly = (c["poly_n"], EPS, LAM)
        s["terms"] = [wd.term(wd.POLY, c["kappa_h"], poly=poly), wd.term(wd.FILTERED, c["kappa_h"], poly=poly),
                      wd.term(wd.HASENBUSCH, c["kappa"], c["kappa_h"])]
        s["params"], s["seed"] = _params(c), int(seed)
    return s


def _as_asked(c, t):
    return t.to(torch.float32) if c["prec"] == "f32" else t


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "batch_cg":
        s["batch"].wd_batch_cg(s["b"], s["x"], s["params"], c["mode"])
        return s["x"]
    lat = s["lat"]
    if kind == "khat":
        lat.mdagm_apply(c["kappa"], PREC[c["prec"]], c["nrhs"], s["in"], s["out"])
        return _as_asked(c, s["out"])
    if kind == "cg":
        s["x"].zero_()
        filt = (c["poly_n"], EPS, LAM) if c["poly_n"] else None
        lat.cg_solve(c["kappa"], s["b"], s["x"], s["params"], filt)
        return s["x"]
    if kind == "force":
        s["F"].zero_()
        lat.fermion_force(s["term"], s["phi"], s["params"], 1.0, s["F"])
        return _as_asked(c, s["F"])
    if kind == "autograd":
        s["w"].grad = None
        S = pf_action(s["w"], lat, s["term"], s["phi"], s["params"], wd.F32)
        S.backward()
        return [S.detach(), _as_asked(c, s["w"].grad)]
    lat.wd_gauge_load(s["U"])
    if kind == "gauge_md":
        s["P"].copy_(s["P0"])
        lat.integrate(s["P"], [], [], [], c["beta"], s["ops"], s["params"], PREC[c["prec"]])
        lat.wd_gauge_store(s["Uout"])
        return [_as_asked(c, s["Uout"]), _as_asked(c, s["P"])]
    p = s["params"]
    r = lat.hmc_trajectory(s["terms"], [1, 0, 0], c["beta"], s["ops"], p, p, wd.F32, s["seed"], 0, 0.0)   # u = 0 accepts
    lat.wd_gauge_store(s["Uout"])
    return [_as_asked(c, s["Uout"]), r["H0"], r["H1"]]


# ---------------------------------------------------------------------------
# work: per site of a half lattice, FP operations of one hop (eight SU(3) x half
# spinor products, projections and sums) and bytes of the inputs and outputs

HOP_FLOPS = 1320


def _khat_flops(vh):
    return 4 * HOP_FLOPS * vh


def _link_bytes(c):
    return 144 if c["prec"] == "f64" else (48 if c.get("recon") else 72)


def work(case):
    c = case
    kind = c["kind"]
    if kind == "batch_cg":
        b = f = 0.0
        for d, n in _batch_groups(c):
            vh = math.prod(d) / 2
            b += n * vh * (8 * 48 + c["nrhs"] * 2 * 192)
            f += n * c["nrhs"] * ITERS * (_khat_flops(vh) + 240 * vh)
        return {"bytes": b, "flops": f}
    vh = math.prod(_dims(c)) / 2
    links = 8 * _link_bytes(c) * vh
    if kind == "khat":
        return {"bytes": links + c["nrhs"] * 2 * 192 * vh, "flops": c["nrhs"] * _khat_flops(vh)}
    if kind == "cg":
        n, k = (ITERS_FILTERED, c["poly_n"] + 1) if c["poly_n"] else (ITERS, 1)
        return {"bytes": links + 2 * 192 * vh, "flops": n * (k * _khat_flops(vh) + 240 * vh)}
    outer = 2 * 4 * (8 * 9 * 2 * 2 + 2 * 198 + 60)           # per output of one (Y, X) pair and half-lattice site
    if kind in ("force", "autograd"):
        n = c["poly_n"]
        solve = {"plain": ITERS, "hasenbusch": ITERS, "poly": 0, "filtered": ITERS_FILTERED * (n + 1)}[c["term"]]
        own = {"plain": 1, "hasenbusch": 2, "poly": 2 * n, "filtered": 2 * n + 2}[c["term"]]
        pairs = {"plain": 1, "hasenbusch": 2, "poly": 2 * n, "filtered": 2 * n + 2}[c["term"]]
        return {"bytes": links + 192 * vh + 512 * vh, "flops": (solve + own) * _khat_flops(vh) + pairs * outer * vh}
    links64 = 8 * 144 * vh
    t_step, g_force = 8 * 1500, 8 * (12 * 198 + 198 + 60)      # per half-lattice site: exponential and product; six staples
    if kind == "gauge_md":
        return {"bytes": 2 * links64 + 2 * 512 * vh, "flops": c["steps"] * (2 * t_step + 2 * g_force) * vh}
    n = c["poly_n"]
    outer_evals = 2 * c["steps"] + 1
    poly_evals = 2 * outer_evals
    k = outer_evals * (ITERS + ITERS_FILTERED * (n + 1) + 2 * n + 4) + poly_evals * 2 * n + 3 * ITERS_FILTERED * (n + 1) + ITERS
    return {"bytes": 2 * links64, "flops": k * _khat_flops(vh) + (4 * poly_evals * (t_step + 2 * g_force)) * vh}


# ---------------------------------------------------------------------------
# the same in 64 bits by plain torch on whole lattices:
# psi [B, R, T, Z, Y, X, 4, 3], links [B, T, Z, Y, X, 4, 3, 3]

# gamma_mu (DeGrand-Rossi): row s holds one entry, _G[mu][s] = (column, value)
_G = [
    [(3, 1j), (2, 1j), (1, -1j), (0, -1j)],
    [(3, -1), (2, 1), (1, 1), (0, -1)],
    [(2, 1j), (3, -1j), (0, -1j), (1, 1j)],
    [(2, 1), (3, 1), (0, 1), (1, 1)],
]


def _gamma(mu, psi):
    perm = [p for p, _ in _G[mu]]
    val = torch.tensor([v for _, v in _G[mu]], dtype=psi.dtype, device=psi.device)
    return psi[..., perm, :] * val[:, None]


def _times(U, psi, dag):
    """U (or U^dag) on the colour index, same links for every right-hand side."""
    if dag:
        return (U.conj().unsqueeze(1).unsqueeze(-3) * psi.unsqueeze(-1)).sum(-2)
    return (U.unsqueeze(1).unsqueeze(-3) * psi.unsqueeze(-2)).sum(-1)


def _hop(U, psi, dag):
    sg = 1.0 if dag else -1.0
    out = 0
    for mu in range(4):
        ax = 5 - mu
        f = torch.roll(psi, -1, ax)
        u = U[..., mu, :, :]
        if mu == 3:
            f = torch.cat([f[:, :, :-1], -f[:, :, -1:]], 2)
        f = _times(u, f, False)
        out = out + f + sg * _gamma(mu, f)
        b = torch.roll(_times(u, psi, True), 1, ax)
        if mu == 3:
            b = torch.cat([-b[:, :, :1], b[:, :, 1:]], 2)
        out = out + b - sg * _gamma(mu, b)
    return out


def _mhat(U, psi, kappa, dag=False):
    return psi - kappa ** 2 * _hop(U, _hop(U, psi, dag), dag)


def _khat(U, psi, kappa):
    return _mhat(U, _mhat(U, psi, kappa), kappa, True)


def _dot(a, b):
    return (a.conj() * b).real.sum(dim=(2, 3, 4, 5, 6, 7), keepdim=True)


def _cg(U, b, kappa, tol=1e-13):
    x, r = torch.zeros_like(b), b.clone()
    p, rr = r.clone(), _dot(r, r)
    stop = tol ** 2 * rr
    for it in range(3000):
        q = _khat(U, p, kappa)
        al = rr / _dot(p, q)
        x, r = x + al * p, r - al * q
        new = _dot(r, r)
        if it % 8 == 7 and bool((new <= stop).all()):
            break
        p = r + (new / rr) * p
        rr = new
    return x


def _poly(U, v, kappa, n):
    """P(K) v, x P(x) = 1 - T_{n+1}((mu - x)/nu) / T_{n+1}(mu/nu)."""
    mu, nu = 0.5 * (LAM + EPS), 0.5 * (LAM - EPS)
    t = [math.cosh(k * math.acosh(mu / nu)) for k in range(n + 2)]
    s0, s1 = torch.zeros_like(v), v / mu
    for k in range(1, n + 1):
        s0, s1 = s1, 2 * t[k] / (nu * t[k + 1]) * (v + mu * s1 - _khat(U, s1, kappa)) - t[k - 1] / t[k + 1] * s0
    return s1


def _even_sites(dims):
    lx, ly, lz, lt = dims
    t, z, y, x = torch.meshgrid(*(torch.arange(n, device="cuda") for n in (lt, lz, ly, lx)), indexing="ij")
    return ((x + y + z + t) % 2 == 0).reshape(-1)


def _to_lex(dims, eo, nr=1):
    """Flat half spinors [nr][12][Vh] -> [1, nr, T, Z, Y, X, 4, 3] (odd sites zero)."""
    lx, ly, lz, lt = dims
    v = lx * ly * lz * lt
    h = torch.view_as_complex(eo.reshape(nr, 12, v // 2, 2)).permute(0, 2, 1)
    out = torch.zeros(nr, v, 12, dtype=torch.complex128, device=eo.device)
    out[:, _even_sites(dims)] = h
    return out.reshape(1, nr, lt, lz, ly, lx, 4, 3)


def _to_eo(dims, psi):
    nr = psi.shape[1]
    h = psi.reshape(nr, -1, 12)[:, _even_sites(dims)].permute(0, 2, 1).contiguous()
    return torch.view_as_real(h).reshape(-1)


def _links_lex(dims, U):
    lx, ly, lz, lt = dims
    return torch.view_as_complex(U.reshape(-1, 2)).reshape(1, lt, lz, ly, lx, 4, 3, 3)


def _alg_to_eo(dims, F):
    """[V, 4, 8] -> flat [4 mu][2 parity][8][Vh]."""
    even = _even_sites(dims)
    return torch.stack([F[even], F[~even]]).permute(2, 0, 3, 1).contiguous().reshape(-1)


def _alg_to_lex(dims, P):
    v = math.prod(dims)
    even = _even_sites(dims)
    h = P.reshape(4, 2, 8, v // 2).permute(1, 3, 0, 2)
    out = torch.empty(v, 4, 8, dtype=torch.float64, device=P.device)
    out[even], out[~even] = h[0], h[1]
    return out


def _force_of(S, U):
    """dS/dw for U -> exp(i w T) U from torch's gradient with respect to U: [V, 4, 8]."""
    (g,) = torch.autograd.grad(S, U)
    W = _mm(U.detach().reshape(-1, 3, 3), g.reshape(-1, 3, 3).mH)
    F = -(W.reshape(-1, 9) @ _T.to(W.device).transpose(-1, -2).reshape(8, 9).T).imag
    return F.reshape(-1, 4, 8)


def _fermion_exact(c, dims, U, phi):
    """(S, force) of one term."""
    kappa, name = c["kappa"], c["term"]
    if name == "poly":
        U.requires_grad_(True)
        S = _dot(phi, _poly(U, phi, kappa, c["poly_n"])).sum()
        return S.detach(), _force_of(S, U)
    psi = _mhat(U, phi, c["kappa_h"], True) if name == "hasenbusch" else phi
    X = _cg(U, psi, kappa)
    S0 = _dot(psi, X).sum()
    U.requires_grad_(True)
    S = -(_mhat(U, X, kappa).abs() ** 2).sum()
    if name == "hasenbusch":
        S = S + 2 * _dot(phi, _mhat(U, X, c["kappa_h"])).sum()
    return S0, _force_of(S, U)


def _gauge_S(U, beta):
    S = 0.0
    for mu in range(4):
        for nu in range(mu + 1, 4):
            um, un = U[..., mu, :, :], U[..., nu, :, :]
            a = _mm(um, torch.roll(un, -1, 4 - mu))
            b = _mm(un, torch.roll(um, -1, 4 - nu))
            S = S + (1.0 - (a * b.conj()).real.sum(dim=(-2, -1)) / 3.0).sum()
    return beta * S


def _gauge_md_exact(c, dims, U, P):
    h = c["tau"] / c["steps"]

    def kick(e):
        nonlocal P
        V = U.clone().requires_grad_(True)
        P = P - e * _force_of(_gauge_S(V, c["beta"]), V)

    def drift(e):
        nonlocal U
        Q = P.reshape(-1, 8)
        flat = U.reshape(-1, 3, 3)
        out = torch.empty_like(flat)
        for s in range(0, flat.shape[0], 1 << 20):
            m = min(flat.shape[0], s + (1 << 20))
            out[s:m] = _mm(_expi(e * _alg(Q[s:m])), flat[s:m])
        U = out.reshape(U.shape)

    for k in range(c["steps"]):
        if k == 0:
            kick(LAM_2MN * h)
        drift(h / 2)
        kick((1 - 2 * LAM_2MN) * h)
        drift(h / 2)
        kick((2 if k + 1 < c["steps"] else 1) * LAM_2MN * h)
    return U, P


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "trajectory" or (kind == "cg" and c["poly_n"]) or c.get("term") == "filtered":
        return None      # a CG of CGs or a chain of them: over the time that is given
    if kind == "batch_cg":
        out, i = [], 0
        ins, kap = _batch_inputs(c, seed), _batch_kappas(c, seed)
        for d, n in _batch_groups(c):
            U = torch.cat([_links_lex(d, u) for _, u, _ in ins[i:i + n]])
            b = torch.cat([_to_lex(d, v, c["nrhs"]) for _, _, v in ins[i:i + n]])
            k = torch.tensor(kap[i:i + n], dtype=torch.float64, device="cuda").reshape(-1, 1, 1, 1, 1, 1, 1, 1)
            x = _cg(U, b, k)
            out += [_to_eo(d, x[j:j + 1]) for j in range(n)]
            i += n
        return out
    dims = _dims(c)
    Uf = _links(dims, c["a"], seed)
    U = _links_lex(dims, Uf)
    half, g = 12 * math.prod(dims), _gen(seed, 1)
    if kind == "khat":
        x = _randn(c["nrhs"] * half, g).reshape(c["nrhs"], -1)
        return torch.cat([_to_eo(dims, _khat(U, _to_lex(dims, v), c["kappa"])) for v in x])
    if kind == "cg":
        return _to_eo(dims, _cg(U, _to_lex(dims, _randn(half, g)), c["kappa"]))
    if kind in ("force", "autograd"):
        S, F = _fermion_exact(c, dims, U.clone(), _to_lex(dims, _randn(half, g)))
        F = _alg_to_eo(dims, F)
        return F if kind == "force" else [S, F]
    P = _alg_to_lex(dims, _randn(32 * math.prod(dims), g))
    V, P = _gauge_md_exact(c, dims, U, P)
    return [torch.view_as_real(V.reshape(-1)).reshape(-1), _alg_to_eo(dims, P)]
