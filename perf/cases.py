"""The library's work as a program gives it, in cases that can be timed and compared.

Six kinds of case, each through the public entry points on device fields:

* ``op``      one application of M^dag M (or of M) by ``lqcd_MdagM`` / ``lqcd_M``: Wilson, domain wall or several
              right-hand sides, FP64, double-float, FP32 or FP16 storage, 12- or 18-real links, the even-odd operator
              or the full one;
* ``force``   the pseudofermion force of one molecular-dynamics step, ``lqcd_force``;
* ``md``      the gauge part of such a step: kinetic energy, gauge force, link update, plaquette;
* ``solve``   a propagator column from the caller's FP64 fields: link and source packing, ``lqcd_eo_solve``, and the
              solution back in the caller's layout;
* ``fields``  a configuration and a propagator taken into the device layout and out of it;
* ``mg``      one multigrid coarse correction: restriction, coarse operator, prolongation.

``exact`` recomputes a case in 64 bits with plain torch operations on the inputs as the device fields hold them.
"""
import math

import torch

import paper_1512_03487_gb300 as L
from paper_1512_03487_gb300 import fields as F

BC = (1.0, 1.0, 1.0, -1.0)
PREC = {"f64": L.LQCD_F64, "f32": L.LQCD_F32, "f16": L.LQCD_F16, "df": L.LQCD_F64_DF}
STORE = {"f64": L.LQCD_F64, "f32": L.LQCD_F32, "f16": L.LQCD_F16, "df": L.LQCD_F64}  # the fields' own format
SUBSET = {"even": L.LQCD_EVEN, "full": L.LQCD_FULL}
SITE_BYTES = {"f64": 192, "f32": 96, "f16": 52, "df": 192}
REAL_BYTES = {"f64": 8, "f32": 4, "f16": 2, "df": 8}
M5, MF = 1.8, 0.02
BETA, MD_STEP = 5.6, 0.05
TOL = 1e-10


# ------------------------------------------------------------------ the cases

def _case(kind, dims, name=None, **kw):
    c = {"kind": kind, "x": dims[0], "y": dims[1], "z": dims[2], "t": dims[3], **kw}
    return {"name": name, **c} if name else c


def _op(dims, prec, recon, subset="even", op="wilson", n5=1, what="MdagM", links="haar", name=None):
    return _case("op", dims, name, prec=prec, recon=recon, subset=subset, op=op, n5=n5, what=what, links=links)


def listed():
    return [
        # the smallest lattice that is used in earnest: four launches, bound by their latency
        _op((8, 8, 8, 8), "f32", 12, name="wilson_f32_8x4"),
        # the inner operator of the headline even-odd solve (FP16 storage, two-row links)
        _op((24, 24, 24, 48), "f16", 12, links="exp", name="wilson_f16_24x48"),
        # the unpreconditioned FP64 operator (the library's defaults) on a lattice whose extents fit no block
        _op((18, 12, 20, 26), "f64", 18, subset="full", name="wilson_f64_full_ragged"),
        # the operator of the solvers' reliable updates, b - M x: double-float arithmetic on the FP64 fields
        _op((24, 24, 24, 48), "df", 18, what="M", links="exp", name="wilson_df_24x48"),
        # domain wall on the paper's 16^4 volume, L_s = 16: the inner operator of that solve
        _op((16, 16, 16, 16), "f32", 12, op="dwf", n5=16, name="dwf_f32_16x4_ls16"),
        # a whole propagator (12 spin-colour columns) at once on 32^4: the largest single operator application
        _op((32, 32, 32, 32), "f16", 12, n5=12, name="wilson_f16_32x4_12rhs"),
        # the fermion force of an HMC step on the larger of the two force lattices
        _case("force", (24, 24, 24, 32), name="force_24x32"),
        # the gauge part of an HMC step on the HMC lattice
        _case("md", (16, 16, 16, 16), name="md_step_16x4"),
        # the headline solve as a program makes it, from its own FP64 fields to the solution in its own layout
        _case("solve", (24, 24, 24, 48), name="solve_f16_24x48", prec="f16", links="exp", mass=0.01),
        # a solve on a small lattice: hundreds of launches of a few microseconds each
        _case("solve", (12, 12, 12, 24), name="solve_f32_12x24", prec="f32", links="haar", mass=0.05),
        # reading a configuration and writing a propagator, extents that fit no block
        _case("fields", (20, 14, 18, 36), name="fields_f32_ragged", prec="f32", recon=12),
        # one coarse correction of the multigrid solver in its usual setting (4^4 aggregates, 12 vectors)
        _case("mg", (24, 24, 24, 48), name="mg_correct_24x48", prec="f32", block=4, nvec=12),
    ]


def _dims(rng, lo, hi, step=2, least=4, most=48):
    """Four extents, multiples of step, whose product is about a log-uniform volume in [lo, hi]."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = v ** 0.25
        d = [max(least, min(most, step * round(side * math.exp(rng.uniform(-0.4, 0.4)) / step))) for _ in range(3)]
        d.append(max(least, min(most, step * round(v / (d[0] * d[1] * d[2]) / step))))
        if 0.7 * lo <= math.prod(d) <= hi:
            return tuple(d)


def draw(rng):
    kind = rng.choice(["op"] * 6 + ["force", "md", "solve", "fields", "mg"])
    if kind == "op":
        op = rng.choice(["wilson", "wilson", "rhs", "dwf"])
        prec = rng.choice(["f64", "f32", "f32", "f16", "f16", "df"])
        recon = rng.choice([12, 18])
        subset = rng.choice(["even", "even", "even", "full"])
        if op == "dwf" and prec == "df":
            recon = 18
        n5 = {"wilson": 1, "rhs": rng.choice([2, 3, 4, 6, 8, 12]), "dwf": rng.choice([8, 16])}[op]
        most = 663552 if prec in ("f64", "df") else 32 ** 4 * (6 if n5 > 1 else 1)
        dims = _dims(rng, 2048, max(4096, most // n5), most=32 if n5 > 1 else 48)
        return _op(dims, prec, recon, subset, "dwf" if op == "dwf" else "wilson", n5,
                   rng.choice(["MdagM", "MdagM", "M"]), rng.choice(["haar", "exp"]))
    if kind == "force":
        return _case("force", _dims(rng, 4096, 442368))
    if kind == "md":
        return _case("md", _dims(rng, 4096, 442368))
    if kind == "solve":
        return _case("solve", _dims(rng, 4096, 131072), prec=rng.choice(["f32", "f16"]),
                     links=rng.choice(["haar", "exp"]), mass=rng.choice([0.05, 0.1]))
    if kind == "fields":
        return _case("fields", _dims(rng, 4096, 663552), prec=rng.choice(["f64", "f32", "f16"]),
                     recon=rng.choice([12, 18]))
    block = rng.choice([2, 4, 4])
    nvec = rng.choice([4, 8, 12, 20]) if block == 4 else rng.choice([3, 4, 6])
    return _case("mg", _dims(rng, 4096, 300000, step=block, least=2 * block), prec="f32", block=block, nvec=nvec)


def _ext(case):
    return case["x"], case["y"], case["z"], case["t"]


def _volume(case):
    return math.prod(_ext(case))


# ------------------------------------------------------------------ inputs (host layouts, complex FP64, on the GPU)

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _gauss(g, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda", dtype=torch.float64))


def _hermitian(g, n):
    """Traceless Hermitian 3x3 matrices (A + A^dag) / 2 - tr / 3 of Gaussian A."""
    a = _gauss(g, n, 3, 3)
    h = 0.5 * (a + a.mH)
    return h - torch.eye(3, dtype=h.dtype, device="cuda") * (h.diagonal(dim1=1, dim2=2).sum(1).real / 3)[:, None, None]


def _su3(a):
    """SU(3) from two independent rows of a: Gram-Schmidt, then the third row."""
    r0 = a[:, 0] / a[:, 0].abs().square().sum(1, keepdim=True).sqrt()
    r1 = a[:, 1] - (r0.conj() * a[:, 1]).sum(1, keepdim=True) * r0
    r1 = r1 / r1.abs().square().sum(1, keepdim=True).sqrt()
    return torch.stack([r0, r1, _row2(r0, r1)], 1)


def _row2(r0, r1):
    return (r0.roll(-1, -1) * r1.roll(-2, -1) - r0.roll(-2, -1) * r1.roll(-1, -1)).conj()


def _links(case, g, kind):
    """U[T, Z, Y, X, mu, 3, 3]: Haar-distributed links ("haar"), or links near exp(0.3 i H) ("exp")."""
    x, y, z, t = _ext(case)
    n = 4 * _volume(case)
    if kind == "haar":
        a = _gauss(g, n, 2, 3)
    else:
        h = 0.3j * _hermitian(g, n)
        a = torch.eye(3, dtype=h.dtype, device="cuda") + h + 0.5 * (h @ h)
    return _su3(a).reshape(t, z, y, x, 4, 3, 3)


def _spinor(case, g, n5=1, subset="full"):
    x, y, z, t = _ext(case)
    return _gauss(g, n5, t, z, y, x // 2 if subset == "even" else x, 4, 3)


# ------------------------------------------------------------------ prepare / run

def _device_spinor(host, lat, prec, subset):
    buf = torch.zeros(L.lqcd_spinor_bytes(lat, prec, subset), dtype=torch.uint8, device="cuda")
    L.lqcd_spinor_pack(buf, prec, subset, torch.view_as_real(host.contiguous()), lat)
    return buf


def _device_links(U, lat, prec, recon):
    buf = torch.zeros(L.lqcd_gauge_bytes(lat, prec, recon), dtype=torch.uint8, device="cuda")
    L.lqcd_gauge_pack(buf, prec, recon, torch.view_as_real(U.contiguous()), lat)
    return buf


def _zeros(nbytes):
    return torch.zeros(nbytes, dtype=torch.uint8, device="cuda")


def _operator(case, prec):
    return L.operator(kind=L.LQCD_DWF if case["op"] == "dwf" else L.LQCD_WILSON, mass=0.01, M5=M5, mf=MF, prec=prec,
                      recon=case["recon"])


def _solver(case):
    return L.solver_params(tol=TOL, maxiter=2000, sloppy_prec=PREC[case["prec"]], sloppy_recon=12, delta=3e-6,
                           delta_mid=0.003 if case["prec"] == "f16" else 0.0, check_interval=64,
                           update_prec=L.LQCD_F64_DF)


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind == "op":
        # links and a spinor in the operator's format, the output field and the operator's workspace
        s["lat"] = lat = L.lattice(_ext(case), n5=case["n5"], bc=BC)
        s["op"] = _operator(case, PREC[case["prec"]])
        store, sub = STORE[case["prec"]], SUBSET[case["subset"]]
        s["links"] = _device_links(_links(case, g, case["links"]), lat, store, case["recon"])
        s["in"] = _device_spinor(_spinor(case, g, case["n5"], case["subset"]), lat, store, sub)
        s["out"] = torch.zeros_like(s["in"])
        s["tmp"] = _zeros(L.lqcd_operator_workspace_bytes(lat, s["op"], sub))
    elif kind == "force":
        # the solution X of M^dag M X = phi stands in as a Gaussian field, Y = M X
        s["lat"] = lat = L.lattice(_ext(case), bc=BC)
        s["op"] = L.operator(mass=0.05)
        s["links"] = _device_links(_links(case, g, "haar"), lat, L.LQCD_F64, 18)
        s["X"] = _device_spinor(_spinor(case, g), lat, L.LQCD_F64, L.LQCD_FULL)
        s["Y"] = torch.zeros_like(s["X"])
        L.lqcd_M(s["Y"], s["X"], s["links"], lat, s["op"], L.LQCD_FULL, 0, None)
        s["out"] = torch.zeros_like(s["links"])
    elif kind == "md":
        s["lat"] = lat = L.lattice(_ext(case), bc=BC)
        s["links"] = _device_links(_links(case, g, "exp"), lat, L.LQCD_F64, 18)
        x, y, z, t = _ext(case)
        s["mom"] = _device_links(_hermitian(g, 4 * _volume(case)).reshape(t, z, y, x, 4, 3, 3), lat, L.LQCD_F64, 18)
        s["out"] = torch.zeros_like(s["links"])
        s["ws"] = _zeros(L.lqcd_reduce_workspace_bytes(lat))
    elif kind == "solve":
        # the caller's own fields, the device fields and the workspace a program keeps between solves
        s["lat"] = lat = L.lattice(_ext(case), bc=BC)
        s["op"], s["prm"] = L.operator(mass=case["mass"]), _solver(case)
        s["U"] = torch.view_as_real(_links(case, g, case["links"]).contiguous())
        s["b"] = torch.view_as_real(_spinor(case, g).contiguous())
        s["x"] = torch.zeros_like(s["b"])
        s["links64"] = _zeros(L.lqcd_gauge_bytes(lat, L.LQCD_F64, 18))
        s["links"] = _zeros(L.lqcd_gauge_bytes(lat, s["prm"].sloppy_prec, 12))
        s["bd"] = _zeros(L.lqcd_spinor_bytes(lat, L.LQCD_F64, L.LQCD_FULL))
        s["xd"] = torch.zeros_like(s["bd"])
        s["ws"] = _zeros(L.lqcd_eo_solve_workspace_bytes(lat, s["op"], s["prm"]))
    elif kind == "fields":
        s["lat"] = lat = L.lattice(_ext(case), bc=BC)
        s["prec"], s["recon"] = PREC[case["prec"]], case["recon"]
        s["U"] = torch.view_as_real(_links(case, g, "haar").contiguous())
        s["b"] = torch.view_as_real(_spinor(case, g).contiguous())
        s["links"] = _zeros(L.lqcd_gauge_bytes(lat, s["prec"], s["recon"]))
        s["bd"] = _zeros(L.lqcd_spinor_bytes(lat, s["prec"], L.LQCD_FULL))
        s["xd"] = _device_spinor(_spinor(case, g), lat, L.LQCD_F64, L.LQCD_FULL)
        s["x"] = torch.zeros_like(s["b"])
    else:
        # orthonormal vectors and a dense coarse stencil; a residual to correct
        s["lat"] = lat = L.lattice(_ext(case), bc=BC)
        vecs, Y, psi = _mg_inputs(case, g)
        prec = PREC[case["prec"]]
        s["vecs"] = torch.cat([_device_spinor(v[None], lat, prec, L.LQCD_FULL) for v in vecs])
        s["Y"], s["psi"] = Y, _device_spinor(psi, lat, prec, L.LQCD_FULL)
        n = Y.shape[1] * Y.shape[2]
        s["c"], s["d"] = (torch.zeros(n, dtype=torch.complex64, device="cuda") for _ in range(2))
        s["out"] = torch.zeros_like(s["psi"])
    return s


def run(s):
    kind, lat = s["kind"], s["lat"]
    if kind == "op":
        sub = SUBSET[s["case"]["subset"]]
        if s["case"]["what"] == "M":
            L.lqcd_M(s["out"], s["in"], s["links"], lat, s["op"], sub, 0, s["tmp"])
        else:
            L.lqcd_MdagM(s["out"], s["in"], s["links"], lat, s["op"], sub, s["tmp"])
        return _typed(s["out"], lat, s["case"]["prec"], s["case"]["subset"])
    if kind == "force":
        L.lqcd_force(s["out"], s["links"], s["X"], s["Y"], lat, s["op"], L.LQCD_FORCE_TA)
        return s["out"].view(torch.float64)
    if kind == "md":
        kin = L.lqcd_momentum_kinetic(s["mom"], lat, s["ws"])
        L.lqcd_gauge_force(s["out"], s["links"], lat, BETA)
        L.lqcd_gauge_exp_update(s["links"], s["mom"], MD_STEP, lat)
        plaq = L.lqcd_plaquette(s["links"], lat, s["ws"])
        return {"force": s["out"].view(torch.float64), "links": s["links"].view(torch.float64), "kinetic": kin,
                "plaquette": plaq}
    if kind == "solve":
        prm = s["prm"]
        L.lqcd_gauge_pack(s["links64"], L.LQCD_F64, 18, s["U"], lat)
        L.lqcd_gauge_pack(s["links"], prm.sloppy_prec, 12, s["U"], lat)
        L.lqcd_spinor_pack(s["bd"], L.LQCD_F64, L.LQCD_FULL, s["b"], lat)
        L.lqcd_eo_solve(s["xd"], s["bd"], s["links64"], s["links"], lat, s["op"], prm, s["ws"])
        L.lqcd_spinor_unpack(s["x"], s["xd"], L.LQCD_F64, L.LQCD_FULL, lat)
        return s["x"]
    if kind == "fields":
        L.lqcd_gauge_pack(s["links"], s["prec"], s["recon"], s["U"], lat)
        L.lqcd_spinor_pack(s["bd"], s["prec"], L.LQCD_FULL, s["b"], lat)
        L.lqcd_spinor_unpack(s["x"], s["xd"], L.LQCD_F64, L.LQCD_FULL, lat)
        return {"links": s["links"].view({"f64": torch.float64, "f32": torch.float32, "f16": torch.float16}[s["case"]["prec"]]),
                "spinor": _typed(s["bd"], lat, s["case"]["prec"], "full"), "host": s["x"]}
    nv, b, prec = s["case"]["nvec"], s["case"]["block"], PREC[s["case"]["prec"]]
    L.lqcd_mg_restrict(s["c"], s["psi"], s["vecs"], nv, b, prec, lat)
    L.lqcd_mg_coarse_apply(s["d"], s["c"], s["Y"], nv, b, prec, 0, lat)
    L.lqcd_mg_prolong(s["out"], s["d"], s["vecs"], nv, b, prec, lat)
    return {"coarse": s["c"], "applied": s["d"], "fine": s["out"].view(torch.float32)}


def _stride(n):
    return (n + 31) // 32 * 32


def _typed(buf, lat, prec, subset):
    """A device spinor field as tensors of its own number types."""
    if prec != "f16":
        return buf.view(torch.float32 if prec == "f32" else torch.float64)
    halves = [buf] if subset == "even" else [buf[: buf.numel() // 2], buf[buf.numel() // 2:]]
    st = halves[0].numel() // 52
    return [{"components": h[: 48 * st].view(torch.float16), "norms": h[48 * st:].view(torch.float32)} for h in halves]


# ------------------------------------------------------------------ work

def work(case):
    v, kind = _volume(case), case["kind"]
    if kind == "op":
        n5, p = case["n5"], case["prec"]
        sites = v * n5 * (1 if case["subset"] == "full" else 0.5)
        hops = (2 if case["subset"] == "even" else 1) * (2 if case["what"] == "MdagM" else 1)
        return {"bytes": 4 * v * case["recon"] * REAL_BYTES[p] + 2 * sites * SITE_BYTES[p], "flops": 1320 * sites * hops}
    if kind == "force":
        return {"bytes": v * (2 * 192 + 4 * 144 * 2), "flops": v * 4 * 826}
    if kind == "md":
        # kinetic: momenta; force: links in, force out; update: links and momenta in, links out; plaquette: links
        return {"bytes": v * 4 * 144 * 3 + v * 4 * 144 * 2, "flops": v * (34 + 4) * 198 + v * 4 * 600}
    if kind == "solve":
        # the FP64 fields in, the solution out; about 60 iterations of four hops over the inner fields
        iters = 60 if case["links"] == "exp" else 24
        per = 4 * (8 * 12 * REAL_BYTES[case["prec"]] + 3 * SITE_BYTES[case["prec"]])
        return {"bytes": v * (4 * 144 + 2 * 192) + iters * v / 2 * per, "flops": iters * v / 2 * 4 * 1320}
    if kind == "fields":
        p = case["prec"]
        return {"bytes": v * (4 * 8 * case["recon"] + 4 * case["recon"] * REAL_BYTES[p] + 192 + SITE_BYTES[p] + 2 * 192),
                "flops": 0}
    nv, vc = case["nvec"], v // case["block"] ** 4
    return {"bytes": v * 96 * (nv + 2) + vc * 8 * (9 * 4 * nv * nv + 4 * nv), "flops": v * 192 * nv + vc * 9 * 4 * nv * nv * 8}


# ------------------------------------------------------------------ the same in 64 bits, with plain torch

def _parity(case):
    x, y, z, t = (torch.arange(n, device="cuda") for n in _ext(case))
    return (t[:, None, None, None] + z[:, None, None] + y[:, None] + x) & 1  # [T, Z, Y, X]


def _to_full(host, case):
    """An even-checkerboard field [n5, T, Z, Y, X/2, ...] on the full lattice, zero on the odd sites."""
    x, y, z, t = _ext(case)
    out = torch.zeros(host.shape[0], t * z * y * x, 4, 3, dtype=host.dtype, device="cuda")
    out[:, (_parity(case) == 0).reshape(-1)] = host.reshape(host.shape[0], -1, 4, 3)
    return out.reshape(-1, t, z, y, x, 4, 3)


def _stored_spinor(psi, prec):
    """psi as a field of this format holds it."""
    if prec in ("f64", "df"):
        return psi
    r = torch.view_as_real(psi).float()
    if prec == "f16":
        m = r.abs().amax(dim=(-3, -2, -1), keepdim=True)
        r = (r * torch.where(m > 0, 1.0 / m, m)).half().double() * m.double()
    return torch.view_as_complex(r.double().contiguous())


def _stored_links(U, prec, recon):
    r = torch.view_as_real(U)
    r = r if prec in ("f64", "df") else r.float().double() if prec == "f32" else r.half().double()
    u = torch.view_as_complex(r.contiguous())
    return u if recon == 18 else torch.cat([u[..., :2, :], _row2(u[..., 0, :], u[..., 1, :])[..., None, :]], -2)


def _B(mu, u0, u1):
    """B_mu applied to a pair of spins: gamma_mu = [[0, B], [B^dag, 0]] in the chiral basis."""
    return ((-1j * u1, -1j * u0), (-u1, u0), (-1j * u0, 1j * u1), (u0, u1))[mu]


def _Bdag(mu, u0, u1):
    return ((1j * u1, 1j * u0), (u1, -u0), (1j * u0, -1j * u1), (u0, u1))[mu]


def _shift(f, mu, d, case, bc=True):
    """f(x + d mu) on [n5, T, Z, Y, X, ...], with the fermions' boundary phase (bc) on the links that wrap."""
    ax = 4 - mu
    out = f.roll(-d, ax)
    if bc and BC[mu] != 1.0:
        out.select(ax, f.shape[ax] - 1 if d > 0 else 0).mul_(BC[mu])
    return out


def _mul(U, h):
    return (U * h.unsqueeze(-2)).sum(-1)


def _hop(U, psi, case, dagger=False):
    """H psi: U [T, Z, Y, X, 4, 3, 3], psi [n5, T, Z, Y, X, 4, 3]."""
    out = torch.zeros_like(psi)
    for mu in range(4):
        u = U[None, ..., mu, :, :]
        for d in (1, -1):
            s = -d if not dagger else d  # forward hop carries (1 - gamma), backward (1 + gamma); dagger swaps
            b0, b1 = _B(mu, psi[..., 2, :], psi[..., 3, :])
            h = [psi[..., 0, :] + s * b0, psi[..., 1, :] + s * b1]
            if d > 0:
                w = [_mul(u, _shift(a, mu, 1, case)) for a in h]
            else:
                w = [_shift(_mul(u.mH, a), mu, -1, case) for a in h]
            l0, l1 = _Bdag(mu, *w)
            out[..., 0, :] += w[0]
            out[..., 1, :] += w[1]
            out[..., 2, :] += s * l0
            out[..., 3, :] += s * l1
    return out


def _m5op(psi, dagger=False):
    """M5op psi(s) = (5 - M5) psi(s) - P_- psi(s + 1) - P_+ psi(s - 1) with mf corners; P_+ on spins 0, 1."""
    up, dn = psi.roll(-1, 0), psi.roll(1, 0)
    up[-1] *= -MF
    dn[0] *= -MF
    if dagger:
        up, dn = dn, up
    out = (5.0 - M5) * psi
    out[..., 2:, :] -= up[..., 2:, :]
    out[..., :2, :] -= dn[..., :2, :]
    return out


def _m5inv(psi, dagger):
    n = psi.shape[0]
    cols = torch.eye(n, dtype=psi.dtype, device="cuda")[:, :, None, None] * torch.ones(4, 1, dtype=psi.dtype, device="cuda")
    m = _m5op(cols, dagger)[..., 0]  # [row s, column s', spin]
    inv = [torch.linalg.inv(m[:, :, 0]), torch.linalg.inv(m[:, :, 2])]
    flat = psi.reshape(n, -1, 4, 3)
    return torch.cat([(inv[c] @ flat[:, :, 2 * c:2 * c + 2].reshape(n, -1)).reshape(n, -1, 2, 3) for c in (0, 1)],
                     2).reshape(psi.shape)


def _apply(case, U, psi, dagger):
    """M psi, or M_hat psi on the even sites of psi (zero on the odd ones)."""
    wilson, c = case["op"] == "wilson", 4.0 + 0.01
    diag = c * psi if wilson else _m5op(psi, dagger)
    h = _hop(U, psi, case, dagger)
    if case["subset"] == "full":
        return diag - 0.5 * h
    h = h / c if wilson else _m5inv(h, dagger)
    return diag - 0.25 * _hop(U, h, case, dagger)


def _chunks(v, per, stride):
    """[n, k] complex site values as the structure of arrays [k / per][stride][per] of a device field."""
    n, k = v.shape
    out = torch.zeros(k // per, stride, per, dtype=v.dtype, device="cuda")
    out[:, :n] = v.reshape(n, k // per, per).transpose(0, 1)
    return torch.view_as_real(out).reshape(-1)


def _layout_spinor(psi, case, prec, subset):
    """psi [n5, T, Z, Y, X, 4, 3] laid out as _typed lays out a device field of this format."""
    par = _parity(case).reshape(-1)
    flat = psi.reshape(psi.shape[0], -1, 12)
    halves = []
    for p in (0,) if subset == "even" else (0, 1):
        v = flat[:, par == p].transpose(0, 1).reshape(-1, 12)
        st = _stride(v.shape[0])
        if prec != "f16":
            halves.append(_chunks(v, 2 if prec == "f32" else 1, st))
            continue
        m = torch.view_as_real(v).abs().amax(dim=(1, 2))
        norms = torch.zeros(st, dtype=torch.float64, device="cuda")
        norms[: m.numel()] = m
        halves.append({"components": _chunks(v / m[:, None], 4, st), "norms": norms})
    return halves if prec == "f16" else torch.cat(halves)


def _layout_links(U, case, prec, recon):
    """U [T, Z, Y, X, 4, 3, 3] in the device layout [parity][mu][chunk][site]."""
    par = _parity(case).reshape(-1)
    flat = U.reshape(-1, 4, 9)[..., : recon // 2]
    st = _stride(_volume(case) // 2)
    per = 1 if prec == "f64" or recon == 18 else 2
    return torch.cat([_chunks(flat[par == p, mu], per, st) for p in (0, 1) for mu in range(4)])


def _exact_op(case, g):
    U = _stored_links(_links(case, g, case["links"]), case["prec"], case["recon"])
    psi = _stored_spinor(_spinor(case, g, case["n5"], case["subset"]), case["prec"])
    if case["subset"] == "even":
        psi = _to_full(psi, case)
    out = _apply(case, U, psi, False)
    if case["what"] == "MdagM":
        out = _apply(case, U, out, True)
    return _layout_spinor(out, case, case["prec"], case["subset"])


def _exact_force(case, g):
    U = _links(case, g, "haar")
    X = _spinor(case, g)
    Y = 4.05 * X - 0.5 * _hop(U, X, case)
    out = torch.zeros_like(U)
    for mu in range(4):
        def proj(p, s):  # (1 + s gamma_mu) p, all four spins
            b, c = _B(mu, p[..., 2, :], p[..., 3, :]), _Bdag(mu, p[..., 0, :], p[..., 1, :])
            return p + s * torch.stack([*b, *c], -2)
        Xn, Yn = _shift(X, mu, 1, case)[0], _shift(Y, mu, 1, case)[0]
        A = (Xn.unsqueeze(-1) * proj(Y[0], -1).conj().unsqueeze(-2)).sum(-3)
        B = (proj(X[0], 1).unsqueeze(-1) * Yn.conj().unsqueeze(-2)).sum(-3)
        u = U[..., mu, :, :]
        G = (u.unsqueeze(-1) * A.unsqueeze(-3)).sum(-2) - (B.unsqueeze(-1) * u.mH.unsqueeze(-3)).sum(-2)
        Fm = 0.5j * (G - G.mH)
        tr = Fm.diagonal(dim1=-2, dim2=-1).sum(-1).real / 3
        out[..., mu, :, :] = Fm - torch.eye(3, dtype=Fm.dtype, device="cuda") * tr[..., None, None]
    return _layout_links(out, case, "f64", 18)


def _mm(a, b):
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _exact_md(case, g):
    x, y, z, t = _ext(case)
    U = _links(case, g, "exp")
    P = _hermitian(g, 4 * _volume(case)).reshape(t, z, y, x, 4, 3, 3)

    def at(V, mu, nu, d):  # V_mu(x + d nu)
        return _shift(V[None, ..., mu, :, :], nu, d, case, bc=False)[0]

    force = torch.zeros_like(U)
    for mu in range(4):
        S = 0
        for nu in range(4):
            if nu == mu:
                continue
            um, un = U[..., mu, :, :], U[..., nu, :, :]
            S = S + _mm(_mm(at(U, nu, mu, 1), at(U, mu, nu, 1).mH), un.mH)
            low = _mm(_mm(um, at(U, nu, mu, 1)).mH, un)  # at x - nu
            S = S + _shift(low[None], nu, -1, case, bc=False)[0]
        W = _mm(U[..., mu, :, :], S)
        Fm = (BETA / 3) * (W - W.mH) / 2j
        tr = Fm.diagonal(dim1=-2, dim2=-1).sum(-1).real / 3
        force[..., mu, :, :] = Fm - torch.eye(3, dtype=Fm.dtype, device="cuda") * tr[..., None, None]
    new = _mm(torch.linalg.matrix_exp((1j * MD_STEP) * P), U)
    plaq = 0.0
    for mu in range(4):
        for nu in range(mu + 1, 4):
            a, b = _mm(new[..., mu, :, :], at(new, nu, mu, 1)), _mm(new[..., nu, :, :], at(new, mu, nu, 1))
            plaq += float((a * b.conj()).real.sum()) / 3
    return {"force": _layout_links(force, case, "f64", 18), "links": _layout_links(new, case, "f64", 18),
            "kinetic": 0.5 * float(P.abs().square().sum()), "plaquette": plaq / (6 * _volume(case))}


def _exact_solve(case, g):
    U = _links(case, g, case["links"])
    b = _spinor(case, g)

    def D(v, dag):
        return (4.0 + case["mass"]) * v - 0.5 * _hop(U, v, case, dag)

    x, r = torch.zeros_like(b), D(b, True)
    p, rr = r.clone(), r.abs().square().sum()
    stop = rr * 1e-30
    for _ in range(1500):
        q = D(D(p, False), True)
        a = rr / (p.conj() * q).sum().real
        x, r = x + a * p, r - a * q
        new = r.abs().square().sum()
        if bool(new < stop):
            break
        p, rr = r + (new / rr) * p, new
    return torch.view_as_real(x)


def _exact_fields(case, g):
    p, recon = case["prec"], case["recon"]
    U = _links(case, g, "haar")
    b, x = _spinor(case, g), _spinor(case, g)
    return {"links": _layout_links(U, case, p, recon), "spinor": _layout_spinor(b, case, p, "full"),
            "host": torch.view_as_real(x)}


def _aggregates(f, case):
    """[..., T, Z, Y, X, 4, 3] as [..., coarse site, chirality, sites * 6]."""
    x, y, z, t = _ext(case)
    b = case["block"]
    f = f.reshape(-1, t // b, b, z // b, b, y // b, b, x // b, b, 2, 2, 3)
    return f.permute(0, 1, 3, 5, 7, 9, 2, 4, 6, 8, 10, 11).reshape(f.shape[0], -1, 2, 6 * b ** 4)


def _from_aggregates(a, case):
    x, y, z, t = _ext(case)
    b = case["block"]
    a = a.reshape(-1, t // b, z // b, y // b, x // b, 2, b, b, b, b, 2, 3)
    return a.permute(0, 1, 6, 2, 7, 3, 8, 4, 9, 5, 10, 11).reshape(-1, t, z, y, x, 4, 3)


def _mg_inputs(case, g):
    """Vectors orthonormal on every aggregate and chirality, a coarse stencil [9][site][Nc][Nc], a fine field."""
    nv = case["nvec"]
    a = _aggregates(torch.cat([_spinor(case, g) for _ in range(nv)]), case)  # [nv, Vc, 2, n]
    a = a.permute(1, 2, 3, 0).contiguous()
    for _ in range(2):  # Cholesky QR, twice: orthonormal to rounding
        ch = torch.linalg.cholesky(a.mH @ a)
        a = torch.linalg.solve_triangular(ch.mH, a, upper=True, left=False)
    vecs = _from_aggregates(a.permute(3, 0, 1, 2), case)
    vc = _volume(case) // case["block"] ** 4
    Y = _gauss(g, 9, vc, 2 * nv, 2 * nv).to(torch.complex64) * (1.0 / math.sqrt(18.0 * nv))
    return vecs, Y, _spinor(case, g)


def _exact_mg(case, g):
    vecs, Y, psi = _mg_inputs(case, g)
    nv, b = case["nvec"], case["block"]
    x, y, z, t = (n // b for n in _ext(case))
    V = _aggregates(_stored_spinor(vecs, case["prec"]), case)                  # [nv, Vc, 2, n]
    f = _aggregates(_stored_spinor(psi, case["prec"]), case)[0]                # [Vc, 2, n]
    c = (V.conj() * f).sum(-1).permute(1, 2, 0).reshape(t, z, y, x, 2 * nv)    # [coarse site][(chirality, k)]
    Yd = Y.to(torch.complex128).reshape(9, t, z, y, x, 2 * nv, 2 * nv)
    d = _mul(Yd[0], c)
    for mu in range(4):
        d = d + _mul(Yd[1 + 2 * mu], c.roll(-1, 3 - mu)) + _mul(Yd[2 + 2 * mu], c.roll(1, 3 - mu))
    out = (V * d.reshape(-1, 2, nv).permute(2, 0, 1).unsqueeze(-1)).sum(0)
    return {"coarse": c.reshape(-1), "applied": d.reshape(-1),
            "fine": _layout_spinor(_from_aggregates(out, case), case, "f32", "full")}


def exact(case, seed):
    g = _gen(seed)
    return {"op": _exact_op, "force": _exact_force, "md": _exact_md, "solve": _exact_solve, "fields": _exact_fields,
            "mg": _exact_mg}[case["kind"]](case, g)
