"""The work that a user of this library has it do, as measurable cases through its public entry points
(`paper_1903_06986_gb300.lqcd`): the Wilson operator in FP64 and in the packed storage of the inner
solver, the Krylov solves, a noise block of a loop estimate, the operator contractions, the HFES
projection on the tensor cores, the exact hopping traces and the link gradient.

Lattices are those of the repository's workloads (4^4, 8^3 x 16, 12^3 x 24, 16^3 x 32, 24^3 x 32) and
ragged ones beside them.  `exact` restates every operation in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

from paper_1903_06986_gb300 import lqcd

EPS = 0.4323        # link width of the repository's synthetic fields (mean plaquette 0.600)
FLAGS = {"M": lqcd.APPLY_M, "Mg5": lqcd.APPLY_G5R, "Mdag": lqcd.APPLY_DAG, "P": lqcd.APPLY_HOP}
PREC = {"f32": lqcd.PREC_F32, "f16": lqcd.PREC_F16, "bf16": lqcd.PREC_BF16}
HALF = {"f16": torch.float16, "bf16": torch.bfloat16}


def _case(kind, dims, **kw):
    return dict(kind=kind, lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3], **kw)


def listed():
    return [
        # one operator application on the paper's smallest lattice: launch latency
        dict(_case("dslash_f64", (4, 4, 4, 4), nrhs=1, flags="M"), name="dslash_f64_4"),
        # the FP64 true residual of a block of ten noises on the largest lattice
        dict(_case("dslash_f64", (24, 24, 24, 32), nrhs=10, flags="Mg5"), name="dslash_f64_24x32"),
        # the inner operator of the mixed-precision noise solves of the same block
        dict(_case("dslash_packed", (24, 24, 24, 32), nrhs=10, flags="Mg5", prec="f16", recon=12),
             name="dslash_f16_24x32"),
        # the same operator with FP32 storage and general links on a ragged lattice, odd block
        dict(_case("dslash_packed", (9, 7, 11, 15), nrhs=3, flags="M", prec="f32", recon=18),
             name="dslash_f32_ragged"),
        # the special right-hand side of a configuration: restarted GMRES-DR(60, 30), FP64
        dict(_case("solve_dr", (8, 8, 8, 16), nrhs=1, m=60, k=30, kappa=0.12), name="solve_dr_8x16"),
        # FP64 noise solves of a block over the deflation space: GMRES-Proj on 50 right-hand sides
        dict(_case("solve_proj", (8, 8, 8, 16), nrhs=50, m=30, k=30, kappa=0.12, system="M", evenodd=False, prec="f64"),
             name="solve_proj_8x16_50"),
        # the same on the even/odd reduced system, one autotuner-sized block
        dict(_case("solve_proj", (12, 12, 12, 24), nrhs=8, m=40, k=40, kappa=0.12, system="Mg5", evenodd=True, prec="f64"),
             name="solve_eo_12x24"),
        # a whole noise block: FP16 inner solves, subtractions, projections, contractions
        dict(_case("noises", (12, 12, 12, 24), nrhs=8, m=40, k=40, kappa=0.12, K=5, npoly=4, prec="f16"),
             name="noises_f16_12x24"),
        # the nine operators of one subtraction mode for a block of ten noises
        dict(_case("contract", (24, 24, 24, 32), nrhs=10, kappa=0.157), name="contract_24x32"),
        # HFES projection over 160 eigenvectors on the tensor cores
        dict(_case("deflate", (16, 16, 16, 32), nrhs=16, k=160, engine="tensor"), name="deflate_tc_16x32"),
        # the exact add-back traces of a configuration's setup (seventh order)
        dict(_case("hop_traces", (8, 8, 8, 16), K=7, kappa=0.157), name="hop_traces_8x16"),
        # the backward pass: link gradient of a block of noises
        dict(_case("link_grad", (12, 12, 12, 24), nrhs=16, kappa=0.155), name="link_grad_12x24"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["dslash_f64", "dslash_packed", "dslash_packed", "solve_dr", "solve_proj", "noises",
                       "contract", "deflate", "hop_traces", "link_grad"])

    def dims(lo, hi, tmax, most, even=False):
        while True:
            d = [_log_int(rng, lo, hi) for _ in range(3)] + [_log_int(rng, lo, tmax)]
            if even:
                d = [x + x % 2 for x in d]
            if d[0] * d[1] * d[2] * d[3] <= most:
                return d

    def block(d, site_rhs, most=16):
        return max(1, min(_log_int(rng, 1, most), site_rhs // (d[0] * d[1] * d[2] * d[3])))

    full = 24 ** 3 * 32
    if kind == "dslash_f64":
        d = dims(4, 24, 32, full)
        return _case(kind, d, nrhs=block(d, 4 * full), flags=rng.choice(sorted(FLAGS)))
    if kind == "dslash_packed":
        d = dims(4, 24, 32, full)
        return _case(kind, d, nrhs=block(d, 10 * full), flags=rng.choice(sorted(FLAGS)),
                     prec=rng.choice(sorted(PREC)), recon=rng.choice([12, 18]))
    if kind == "solve_dr":
        k = rng.randint(5, 30)
        return _case(kind, dims(4, 10, 16, 8 ** 3 * 16), nrhs=1, m=k + rng.randint(10, 30), k=k,
                     kappa=round(rng.uniform(0.11, 0.12), 4))
    if kind == "solve_proj":
        eo = rng.random() < 0.3
        d = dims(4, 12, 24, 8 ** 3 * 16, even=eo)
        return _case(kind, d, nrhs=_log_int(rng, 1, 32), m=rng.randint(15, 40), k=rng.randint(5, 30),
                     kappa=round(rng.uniform(0.11, 0.12), 4), system=rng.choice(["M", "Mg5"]), evenodd=eo,
                     prec="f64" if eo else rng.choice(["f64", "f32", "f16", "bf16"]))
    if kind == "noises":
        return _case(kind, rng.choice([(8, 8, 8, 8), (6, 6, 6, 12), (6, 12, 6, 12), (12, 12, 12, 12)]),
                     nrhs=rng.randint(2, 12), m=rng.randint(20, 40), k=rng.randint(5, 40),
                     kappa=round(rng.uniform(0.11, 0.12), 4), K=rng.randint(3, 5), npoly=rng.randint(2, 4),
                     prec=rng.choice(["f64", "f32", "f16", "bf16"]))
    if kind == "contract":
        d = dims(4, 24, 32, full)
        return _case(kind, d, nrhs=block(d, 8 * full, 60), kappa=round(rng.uniform(0.12, 0.16), 4))
    if kind == "deflate":
        d = dims(4, 16, 32, 16 ** 3 * 32)
        return _case(kind, d, nrhs=rng.randint(1, 16), k=_log_int(rng, 4, 160),
                     engine="tensor" if d[0] * d[1] * d[2] * d[3] > 20000 else rng.choice(["tensor", "f64"]))
    if kind == "hop_traces":
        d, kmax = rng.choice([((4, 4, 4, 8), 7), ((4, 6, 8, 4), 5), ((6, 6, 6, 12), 5), ((8, 8, 8, 8), 7),
                              ((5, 4, 3, 6), 6)])
        return _case(kind, d, K=rng.randint(min(5, kmax), kmax), kappa=round(rng.uniform(0.12, 0.16), 4))
    d = dims(4, 16, 32, 12 ** 3 * 24)
    return _case(kind, d, nrhs=rng.randint(1, 16), kappa=round(rng.uniform(0.12, 0.16), 4))


# ---- inputs ---------------------------------------------------------------------------------------
def _dims(c):
    return c["lx"], c["ly"], c["lz"], c["lt"]


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _gauss(g, shape):
    return torch.complex(torch.randn(shape, generator=g, device="cuda", dtype=torch.float64),
                         torch.randn(shape, generator=g, device="cuda", dtype=torch.float64))


def _links(c, g):
    """Near-identity SU(3) links exp(i EPS H), H traceless Hermitian Gaussian (as synth.su3_links)."""
    lx, ly, lz, lt = _dims(c)
    A = _gauss(g, (4 * lt * lz * ly * lx, 3, 3)) / math.sqrt(2.0)
    H = 0.5 * (A + A.mH)
    eye = torch.eye(3, dtype=A.dtype, device=A.device)
    H = 1j * EPS * (H - (H.diagonal(dim1=-2, dim2=-1).sum(-1) / 3.0)[:, None, None] * eye)
    U, term = eye + H, H
    for j in range(2, 24):
        term = (term[:, :, :, None] * H[:, None, :, :]).sum(2) / j
        U = U + term
    r1 = U[:, 0] / torch.linalg.vector_norm(U[:, 0], dim=-1, keepdim=True)
    r2 = U[:, 1] - (r1.conj() * U[:, 1]).sum(-1, keepdim=True) * r1
    r2 = r2 / torch.linalg.vector_norm(r2, dim=-1, keepdim=True)
    r3 = torch.linalg.cross(r1, r2, dim=-1).conj()
    return torch.stack([r1, r2, r3], dim=1).reshape(4, lt, lz, ly, lx, 3, 3).contiguous()


def _field(c, g, n):
    lx, ly, lz, lt = _dims(c)
    return _gauss(g, (n, lt, lz, ly, lx, 4, 3))


def _unit(f):
    flat = f.reshape(f.shape[0], -1)
    return (flat / torch.linalg.vector_norm(flat, dim=1, keepdim=True)).reshape(f.shape)


def _noise(seed, first, c, n):
    """Z(4) noises (Philox-4x32-10, key = seed, counter = (noise, site, 0, 0)), restated in numpy."""
    lx, ly, lz, lt = _dims(c)
    V = lx * ly * lz * lt
    m32 = np.uint64(0xFFFFFFFF)
    c0 = np.repeat(np.arange(first, first + n, dtype=np.uint64), V)
    c1 = np.tile(np.arange(V, dtype=np.uint64), n)
    c2, c3 = np.zeros_like(c0), np.zeros_like(c0)
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c0, np.uint64(0xCD9E8D57) * c2
        c0, c1, c2, c3 = ((p1 >> np.uint64(32)) ^ c1 ^ np.uint64(k0), p1 & m32,
                          (p0 >> np.uint64(32)) ^ c3 ^ np.uint64(k1), p0 & m32)
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    code = (c0[:, None] >> (2 * np.arange(12, dtype=np.uint64))) & np.uint64(3)
    z = np.array([1, 1j, -1, -1j], dtype=np.complex128)[code.astype(np.int64)]
    return torch.from_numpy(z.reshape(n, lt, lz, ly, lx, 4, 3)).cuda()


def _noise_seed(seed):
    return 1000003 * (seed % (1 << 40)) + 17


def _poly(n):
    """a_j of the truncated Neumann polynomial sum_{i<=n} (1 - M)^i (saved POLY coefficients)."""
    return np.array([(-1.0) ** j * math.comb(n + 1, j + 1) for j in range(n + 1)], dtype=np.complex128)


def _eigen(c, g, k):
    """Unit fields and eigenvalues standing for saved eigenpairs of M gamma_5."""
    E = _unit(_field(c, g, k))
    sign = np.where(np.arange(k) % 2 == 0, 1.0, -1.0)
    return E, (sign * np.linspace(0.05, 0.6, k)).astype(np.complex128)


def prepare(case, seed):
    c, g, kind = case, _gen(seed), case["kind"]
    s = dict(case=c, kind=kind)
    if kind != "deflate":
        s["U"] = _links(c, g)
    recon = 12 if kind == "noises" else 18
    ctx = s["ctx"] = (lqcd.EvenOddContext(_dims(c)) if c.get("evenodd") else lqcd.Context(_dims(c), recon=recon))
    if kind == "dslash_f64":
        s["in"] = _field(c, g, c["nrhs"])
        s["out"] = torch.empty_like(s["in"])
    elif kind == "dslash_packed":
        f = _unit(_field(c, g, c["nrhs"]))
        s["Up"] = ctx.pack_links_f32(s["U"], c["recon"])
        s["in"] = ctx.pack_f32(f) if c["prec"] == "f32" else ctx.pack_half(f, PREC[c["prec"]])
        s["out"] = torch.empty_like(s["in"])
    elif kind == "solve_dr":
        s["b"] = _noise(_noise_seed(seed), 0, c, 1)
    elif kind == "solve_proj":
        nz = _noise(_noise_seed(seed), 0, c, c["nrhs"] + 1)
        if c["evenodd"]:
            nz = torch.cat([ctx.rhs(s["U"], c["kappa"], nz[i:i + 1].contiguous()) for i in range(nz.shape[0])])
        s["b"] = nz[:-1].contiguous()
        solve = ctx.gmresdr_solve if c["system"] == "M" else ctx.minresdr_solve
        s["defl"] = solve(s["U"], c["kappa"], nz[-1:].contiguous(), c["k"] + 20, c["k"], 1e-3, max_cycles=3,
                          want_defl=True)[2]
    elif kind == "noises":
        b = _noise(_noise_seed(seed), 0xFFFFFFFE, c, 1)
        proj = ctx.minresdr_solve(s["U"], c["kappa"], b, c["k"] + 20, c["k"], 1e-3, max_cycles=3, want_defl=True)[2]
        E, lam = _eigen(c, g, c["k"])
        ctx.set_defl_engine(lqcd.DEFL_TENSOR)
        ctx.set_inner_window(2)
        s["loop"] = ctx.loop_setup_from(
            s["U"], c["kappa"], proj, ctx.defl_import(E, lam), _poly(c["npoly"]), _noise_seed(seed), c["nrhs"],
            c["nrhs"], c["k"] + 20, c["k"], c["K"], c["npoly"], 1e-12, 1e-3, m_inner=c["m"],
            modes=lqcd.SUB_ALL & ~lqcd.SUB_ES, prec=PREC.get(c["prec"], lqcd.PREC_F64), inner_tol=0.1,
            system=lqcd.SYS_MG5)
    elif kind == "contract":
        # a noise block and its solution-like partner
        s["eta"] = _noise_like(g, _field(c, g, c["nrhs"]))
        s["w"] = s["eta"] + 0.3 * _field(c, g, c["nrhs"])
    elif kind == "deflate":
        E, lam = _eigen(c, g, c["k"])
        s["defl"] = ctx.defl_import(E, lam)
        s["d"] = 1.0 / lam
        s["eta"] = _noise_like(g, _field(c, g, c["nrhs"]))
        ctx.set_defl_engine(lqcd.DEFL_TENSOR if c["engine"] == "tensor" else lqcd.DEFL_FP64)
    elif kind == "link_grad":
        s["z"], s["x"] = _field(c, g, c["nrhs"]), _field(c, g, c["nrhs"])
    return s


def _noise_like(g, f):
    """Z(4)-valued field of the shape of f."""
    code = torch.randint(0, 4, f.shape, generator=g, device="cuda")
    return torch.tensor([1, 1j, -1, -1j], dtype=torch.complex128, device="cuda")[code]


def run(state):
    s, c, ctx = state, state["case"], state["ctx"]
    kind = s["kind"]
    if kind == "dslash_f64":
        return ctx.wilson_apply(s["U"], 0.157, s["in"], out=s["out"], flags=FLAGS[c["flags"]])
    if kind == "dslash_packed":
        if c["prec"] == "f32":
            return ctx.wilson_apply_packed(s["Up"], c["recon"], 0.157, s["in"], out=s["out"], flags=FLAGS[c["flags"]])
        return ctx.wilson_apply_half(s["Up"], c["recon"], 0.157, s["in"], out=s["out"], flags=FLAGS[c["flags"]],
                                     prec=PREC[c["prec"]]).view(HALF[c["prec"]])
    if kind == "solve_dr":
        return ctx.gmresdr_solve(s["U"], c["kappa"], s["b"], c["m"], c["k"], 1e-12)[0]
    if kind == "solve_proj":
        return ctx.proj_solve(s["U"], c["kappa"], s["defl"], s["b"], c["m"], 1e-12,
                              prec=PREC.get(c["prec"], lqcd.PREC_F64))[0]
    if kind == "noises":
        return s["loop"].noises(s["U"], 0, c["nrhs"])[0]
    if kind == "contract":
        return ctx.contract(s["U"], c["kappa"], s["eta"], s["w"])
    if kind == "deflate":
        return ctx.deflate_project(s["defl"], s["eta"], s["d"])
    if kind == "hop_traces":
        return ctx.hop_traces(s["U"], c["kappa"], c["K"])
    return lqcd.link_grad(ctx, s["U"], c["kappa"], s["z"], s["x"])


# ---- work a pass cannot do without ------------------------------------------------------------------
def work(case):
    c, kind = case, case["kind"]
    V = c["lx"] * c["ly"] * c["lz"] * c["lt"]
    n = c.get("nrhs", 1)
    fld, lnk, dsl = 192.0 * V, 576.0 * V, 1368.0 * V     # bytes of an FP64 field and of the links; flops of M
    if kind == "dslash_f64":
        return dict(bytes=2 * n * fld + lnk, flops=n * dsl)
    if kind == "dslash_packed":
        size = 4 if c["prec"] == "f32" else 2
        return dict(bytes=48.0 * V * size * n + 16.0 * V * 4 * (3 if c["recon"] == 12 else 5), flops=n * dsl)
    if kind in ("solve_dr", "solve_proj", "noises"):
        # applications to 1e-12 at these kappa (M gamma_5 is indefinite and takes more), each new basis
        # vector orthogonalised against the ones before it (one pass of inner products and updates;
        # two of them in the Lanczos recurrence of the noise block)
        it, half = 450 if kind == "noises" else 90 if c.get("system", "M") == "M" else 400, 1
        if c.get("evenodd"):
            it, half = it * 2 // 5, 2
        vec = 2 if kind == "noises" else min(it, c["m"]) / 2
        size = {"f64": 1.0, "f32": 0.5, "f16": 0.25, "bf16": 0.25}[c.get("prec", "f64")]
        w = dict(bytes=it * (n * (3 + vec) * fld * size / half + lnk * size),
                 flops=it * n * (dsl + 16 * 12.0 * V * vec / half))
        if kind == "noises":
            w["bytes"] += n * 20 * fld + 2 * c["k"] * fld
            w["flops"] += n * ((c["K"] - 1 + c["npoly"] + 6 * 2) * dsl + 3 * 16 * 12.0 * V * c["k"])
        return w
    if kind == "contract":
        return dict(bytes=2 * n * fld + lnk, flops=n * V * 2000.0)
    if kind == "deflate":
        return dict(bytes=(c["k"] + 2 * n) * fld, flops=16.0 * 12 * V * c["k"] * n)
    if kind == "hop_traces":
        ncls = min(2.0 * ((c["K"] + 2) // 2) ** 4, V)
        return dict(bytes=12 * ncls * (c["K"] - 1) * fld / 2, flops=12 * ncls * (c["K"] - 1) / 2 * dsl)
    return dict(bytes=2 * n * fld + lnk + 4 * V * 17 * 16.0, flops=n * 4 * V * 1500.0)


# ---- the same in 64 bits with plain torch -------------------------------------------------------------
_AXIS = {0: 4, 1: 3, 2: 2, 3: 1}     # lattice axis of direction mu in a (n, T, Z, Y, X, 4, 3) field


def _gammas():
    s = [np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]])]
    o = np.zeros((2, 2))
    g = [np.block([[o, -1j * a], [1j * a, o]]) for a in s] + [np.diag([1, 1, -1, -1])]
    g5 = g[0] @ g[1] @ g[2] @ g[3]
    dev = lambda a: torch.tensor(a, dtype=torch.complex128, device="cuda")
    return [dev(a) for a in g], dev(g5)


def _spin(a, p):
    """(a p) for a 4 x 4 spin matrix."""
    rows = []
    for i in range(4):
        acc = torch.zeros_like(p[..., 0, :])
        for j in range(4):
            if a[i, j] != 0:
                acc = acc + a[i, j] * p[..., j, :]
        rows.append(acc)
    return torch.stack(rows, dim=-2)


def _col(u, p):
    """U p for links u (..., 3, 3) and spinors p (n, ..., 4, 3)."""
    return sum(u[..., None, :, b] * p[..., b, None] for b in range(3))


def _hop(U, p):
    gam, _ = _gammas()
    one = torch.eye(4, dtype=torch.complex128, device="cuda")
    out = torch.zeros_like(p)
    for mu in range(4):
        ax = _AXIS[mu]
        out += _col(U[mu], _spin(one - gam[mu], torch.roll(p, -1, ax)))
        out += torch.roll(_col(U[mu].mH, _spin(one + gam[mu], p)), 1, ax)
    return out


def _g5(p):
    return _spin(_gammas()[1], p)


def _wilson(U, kappa, p, flags="M"):
    if flags == "P":
        return _hop(U, p)
    q = _g5(p) if flags in ("Mg5", "Mdag") else p
    r = q - kappa * _hop(U, q)
    return _g5(r) if flags == "Mdag" else r


def _solve(U, kappa, b):
    """M x = b to rounding: conjugate gradients on M^dag M with one correction from the true residual."""
    dot = lambda u, v: (u.conj() * v).real.flatten(1).sum(1).reshape(-1, *([1] * (b.dim() - 1)))
    x = torch.zeros_like(b)
    for _ in range(3):
        res = b - _wilson(U, kappa, x)
        r = _wilson(U, kappa, res, "Mdag")
        p, rr = r.clone(), dot(r, r)
        stop, d = rr.max().item() * 1e-26, torch.zeros_like(b)
        for it in range(1500):
            q = _wilson(U, kappa, p)
            a = rr / dot(q, q).clamp_min(1e-300)
            d += a * p
            r = r - a * _wilson(U, kappa, q, "Mdag")
            new = dot(r, r)
            p, rr = r + new / rr.clamp_min(1e-300) * p, new
            if it % 10 == 9 and rr.max().item() < stop:
                break
        x = x + d
    return x


def _contract(U, kappa, eta, w):
    """(n, 9, T) densities of eta^dag Theta w summed per timeslice."""
    gam, _ = _gammas()
    one = torch.eye(4, dtype=torch.complex128, device="cuda")
    dens = lambda a, b: (a.conj() * b).sum(dim=(2, 3, 4, 5, 6))
    ops = [dens(eta, w)] + [dens(eta, _spin(gam[mu], w)) for mu in range(4)]
    for mu in range(4):
        ax = _AXIS[mu]
        fwd = dens(torch.roll(eta, -1, ax), _spin(one + gam[mu], _col(U[mu].mH, w)))
        bwd = dens(eta, _spin(one - gam[mu], _col(U[mu], torch.roll(w, -1, ax))))
        ops.append(kappa * (fwd - bwd))
    return torch.stack(ops, dim=1)


def _deflate(E, d, eta):
    flat, out = E.reshape(E.shape[0], -1), []
    d = torch.as_tensor(d, device="cuda")
    for i in range(eta.shape[0]):
        co = (flat.conj() @ eta[i].reshape(-1)) * d
        out.append((co @ flat).reshape(eta.shape[1:]))
    return _g5(torch.stack(out))


def _pack(p):
    """canonical (n, T, Z, Y, X, 4, 3) -> the packed chunk-major order, as reals (n, 24 V)."""
    q = p.reshape(p.shape[0], -1, 6, 2).permute(0, 2, 1, 3).contiguous()
    return torch.view_as_real(q).reshape(p.shape[0], -1)


def _unpack(c, x):
    lx, ly, lz, lt = _dims(c)
    q = torch.view_as_complex(x.double().reshape(x.shape[0], 6, -1, 2, 2).contiguous())
    return q.permute(0, 2, 1, 3).reshape(x.shape[0], lt, lz, ly, lx, 4, 3)


def _parity(c):
    lx, ly, lz, lt = _dims(c)
    r = [torch.arange(v, device="cuda") for v in (lt, lz, ly, lx)]
    return (r[0][:, None, None, None] + r[1][:, None, None] + r[2][:, None] + r[3]) % 2


def _traces(c, U):
    """Exact hopping traces by probing the classes (x mod s, ..., sum floor(x / s) mod 2), s = ceil((K + 1) / 2):
    members more than K hops apart where 2 s divides every extent; None on other lattices."""
    dims, K = _dims(c), c["K"]
    st = (K + 2) // 2
    if any(d % (2 * st) for d in dims):
        return None
    gam, _ = _gammas()
    one = torch.eye(4, dtype=torch.complex128, device="cuda")
    lx, ly, lz, lt = dims
    co = torch.stack(torch.meshgrid(*(torch.arange(v, device="cuda") for v in (lt, lz, ly, lx)), indexing="ij")[::-1])
    res, cell = co % st, (co // st).sum(0) % 2
    cls = (cell + 2 * (res[0] + st * (res[1] + st * (res[2] + st * res[3])))).reshape(-1)
    V = lx * ly * lz * lt
    site = torch.arange(V, device="cuda").reshape(lt, lz, ly, lx)
    nxt = [torch.roll(site, -1, 3 - mu).reshape(-1) for mu in range(4)]
    prv = [torch.roll(site, 1, 3 - mu).reshape(-1) for mu in range(4)]
    tim = co[3].reshape(-1)
    Uf = U.reshape(4, V, 3, 3)
    out = torch.zeros((K, 9, lt), dtype=torch.complex128, device="cuda")
    tr = lambda m: m.diagonal(dim1=0, dim2=2).sum(-1)     # (12, members, 12) -> trace per member
    step = max(1, 16384 * 12 // (12 * V))
    eye = torch.eye(12, dtype=torch.complex128, device="cuda")
    for c0 in range(0, 2 * st ** 4, step):
        mem = [torch.nonzero(cls == k).reshape(-1) for k in range(c0, min(c0 + step, 2 * st ** 4))]
        z = torch.zeros((len(mem) * 12, V, 12), dtype=torch.complex128, device="cuda")
        for i, m in enumerate(mem):
            z[12 * i:12 * i + 12, m] = eye[:, None, :]
        w = z.reshape(-1, lt, lz, ly, lx, 4, 3)
        for k in range(K):
            if k:
                w = _hop(U, w)
            for i, m in enumerate(mem):
                wi = w[12 * i:12 * i + 12].reshape(12, V, 4, 3)
                at = lambda a: a.reshape(12, -1, 12)
                out[k, 0].index_add_(0, tim[m], tr(at(wi[:, m])))
                for mu in range(4):
                    out[k, 1 + mu].index_add_(0, tim[m], tr(at(_spin(gam[mu], wi[:, m]))))
                    b = prv[mu][m]
                    t1 = _spin(one + gam[mu], _col(Uf[mu][b].mH, wi[:, b]))
                    t2 = _spin(one - gam[mu], _col(Uf[mu][m], wi[:, nxt[mu][m]]))
                    out[k, 5 + mu].index_add_(0, tim[b], c["kappa"] * tr(at(t1)))
                    out[k, 5 + mu].index_add_(0, tim[m], -c["kappa"] * tr(at(t2)))
    return out


def _gell_mann():
    l = np.zeros((8, 3, 3), dtype=np.complex128)
    l[0][0, 1] = l[0][1, 0] = 1
    l[1][0, 1], l[1][1, 0] = -1j, 1j
    l[2][0, 0], l[2][1, 1] = 1, -1
    l[3][0, 2] = l[3][2, 0] = 1
    l[4][0, 2], l[4][2, 0] = -1j, 1j
    l[5][1, 2] = l[5][2, 1] = 1
    l[6][1, 2], l[6][2, 1] = -1j, 1j
    l[7] = np.diag([1, 1, -2]) / math.sqrt(3.0)
    return torch.tensor(l, device="cuda")


def _link_grad(U, kappa, z, x):
    gam, _ = _gammas()
    one = torch.eye(4, dtype=torch.complex128, device="cuda")
    lam = _gell_mann()
    outer = lambda a, b: sum(a[..., s, :, None] * b[..., s, None, :] for s in range(4)).sum(0)
    g, gl = [], []
    for mu in range(4):
        xf, zf = torch.roll(x, -1, _AXIS[mu]), torch.roll(z, -1, _AXIS[mu])
        pm, pp = _spin(one - gam[mu], xf), _spin(one + gam[mu], x)
        B = outer(_col(U[mu], pm), z.conj()) - outer(pp, _col(U[mu], zf).conj())
        g.append(0.5j * kappa * torch.einsum("acd,...dc->...a", lam, B))
        dU, dUc = kappa * outer(z.conj(), pm), kappa * outer(pp, zf.conj())
        gl.append(dUc + dU.conj())
    return torch.stack(g), torch.stack(gl)


def exact(case, seed):
    c, g, kind = case, _gen(seed), case["kind"]
    U = _links(c, g) if kind != "deflate" else None
    if kind == "dslash_f64":
        f = _field(c, g, c["nrhs"])
        return torch.cat([_wilson(U, 0.157, f[i:i + 1], c["flags"]) for i in range(c["nrhs"])])
    if kind == "dslash_packed":
        f = _unit(_field(c, g, c["nrhs"]))
        n = f[0].numel()
        if c["prec"] == "f32":
            f = _unpack(c, _pack(f).float())
        else:
            f = _unpack(c, (_pack(f) * 2.0 ** math.floor(0.5 * math.log2(n))).to(HALF[c["prec"]]))
        return torch.cat([_pack(_wilson(U, 0.157, f[i:i + 1], c["flags"])) for i in range(c["nrhs"])])
    if kind == "solve_dr":
        return _solve(U, c["kappa"], _noise(_noise_seed(seed), 0, c, 1))
    if kind == "solve_proj":
        b = _noise(_noise_seed(seed), 0, c, c["nrhs"])
        x = _solve(U, c["kappa"], b)
        if c["system"] == "Mg5":
            x = _g5(x)              # a space of M gamma_5: the solve is M gamma_5 y = b
        if c["evenodd"]:            # the even sites of the full solution solve the reduced system
            x = x.reshape(c["nrhs"], -1, 4, 3)[:, (_parity(c) == 0).reshape(-1)]
        return x
    if kind == "noises":
        k, kappa, nz = c["k"], c["kappa"], c["nrhs"]
        E, lam = _eigen(c, g, k)
        eta = _noise(_noise_seed(seed), 0, c, nz)
        x = _solve(U, kappa, eta)
        a = _poly(c["npoly"])

        def pert(v):
            out, t = v.clone(), v
            for _ in range(1, c["K"]):
                t = kappa * _hop(U, t)
                out += t
            return out

        def poly(v):
            out, t = a[0].item() * v, v
            for j in range(1, len(a)):
                t = _wilson(U, kappa, t)
                out = out + a[j].item() * t
            return out

        def xi(f):
            return np.array([torch.vdot(e.reshape(-1), _g5(f(e[None])).reshape(-1)).item() for e in E])

        xp, xq, none = pert(eta), poly(eta), torch.zeros_like(eta)
        sub = [none, xp, xq, _deflate(E, 1 / lam, eta), xp + _deflate(E, 1 / lam - xi(pert), eta),
               xq + _deflate(E, 1 / lam - xi(poly), eta)]
        out = [_contract(U, kappa, eta, x - v) for v in sub]
        return torch.stack(out + [torch.zeros_like(out[0])]).cpu().numpy()
    if kind == "contract":
        eta = _noise_like(g, _field(c, g, c["nrhs"]))
        w = eta + 0.3 * _field(c, g, c["nrhs"])
        return torch.cat([_contract(U, c["kappa"], eta[i:i + 1], w[i:i + 1]) for i in range(c["nrhs"])]).cpu().numpy()
    if kind == "deflate":
        E, lam = _eigen(c, g, c["k"])
        return _deflate(E, 1.0 / lam, _noise_like(g, _field(c, g, c["nrhs"])))
    if kind == "hop_traces":
        t = _traces(c, U)
        return None if t is None else t.cpu().numpy()
    z, x = _field(c, g, c["nrhs"]), _field(c, g, c["nrhs"])
    return _link_grad(U, c["kappa"], z, x)
