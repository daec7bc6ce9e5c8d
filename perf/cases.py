"""The calls whose speed is measured: what a lattice-QCD user of this package spends time on.

Each case is one pass through the public binding (paper_0905_3331_gb300.tm) on device buffers:

  hop       H_eo / H_oe on stacked half fields (Lattice.apply_hopping_eo), in the storage forms that
            the solvers and the benchmark use
  dirac     the full operator M or M^dag on canonical FP64 fields (Lattice.apply_D)
  fields    canonical half fields to a device storage form and back (pack_half, unpack_half)
  solve     one solve M x = b of a Gaussian source, mixed precision (Lattice.solve_cg)
  normal    the FP64 solve of the normal equations that a pseudofermion force needs (solve_normal)
  points    the twelve point sources of a propagator in one batched solve (solve_cg_batch)
  contract  timeslice Gram matrices of a propagator and three correlators (meson_contract, correlator)

The gauge fields are random SU(3) links U = exp(i eps H) as in the package's own synthetic inputs, with
the eps, kappa and mu of its workloads (4^4 to 48^3 x 96); sources are Gaussian or point sources; the
propagators of the contraction are Gaussian with an exponential decay in time.  `exact` evaluates the
same passes with plain torch in complex128.
"""
import math

import numpy as np
import torch

from paper_0905_3331_gb300 import tm

F64, F32, F16 = tm.F64, tm.F32, tm.F16
PREC = {"f64": F64, "f32": F32, "f16": F16}


def listed():
    return [
        # the smallest lattice of the workloads: one launch, nothing but latency
        dict(name="hop_f64_4x4", kind="hop", T=4, L=4, prec="f64", link=18, parity=1, nrhs=1),
        # the full operator on a small lattice: several launches of almost no work
        dict(name="dirac_8x8", kind="dirac", T=8, L=8, nrhs=1, flavour=1, dagger=False),
        # M^dag of the other flavour on two fields, extents that divide no tile
        dict(name="dirac_dag_14x20", kind="dirac", T=20, L=14, nrhs=2, flavour=-1, dagger=True),
        # the full operator on a production lattice (residual checks, measurements)
        dict(name="dirac_32x64", kind="dirac", T=64, L=32, nrhs=1, flavour=1, dagger=False),
        # the sloppy operator of a 16^3 x 32 solve
        dict(name="hop_f32_16x32", kind="hop", T=32, L=16, prec="f32", link=12, parity=0, nrhs=1),
        # several right-hand sides with half-precision storage
        dict(name="hop_f16_24x48_n4", kind="hop", T=48, L=24, prec="f16", link=12, parity=1, nrhs=4),
        # the sloppy operator of the headline solve on the largest lattice
        dict(name="hop_f16_48x96", kind="hop", T=96, L=48, prec="f16", link=8, parity=0, nrhs=1),
        # a caller's fields into the FP32 storage form and back, as around every use of half fields
        dict(name="fields_f32_24x48", kind="fields", T=48, L=24, prec="f32", nrhs=2),
        # one propagator column, mixed precision
        dict(name="solve_f32_16x32", kind="solve", T=32, L=16, prec="f32", link=12, delta=1e-5, upd="f64"),
        # FP64 normal equations (the heat-bath and force solves of an HMC trajectory)
        dict(name="normal_f64_12x24", kind="normal", T=24, L=12),
        # a whole propagator: twelve point sources at once
        dict(name="points_f32_16x32", kind="points", T=32, L=16, prec="f32", link=12, delta=1e-3),
        # its meson correlators on a production lattice
        dict(name="contract_24x48", kind="contract", T=48, L=24),
    ]


def draw(rng):
    kind = rng.choice(["hop", "hop", "hop", "dirac", "dirac", "fields", "solve", "normal", "contract"])
    most = {"hop": 48 ** 3 * 96, "dirac": 32 ** 3 * 64, "fields": 24 ** 3 * 48 * 2, "solve": 16 ** 3 * 32,
            "normal": 12 ** 3 * 24, "contract": 24 ** 3 * 48}[kind]
    least = 2048 if kind in ("solve", "normal") else 256
    while True:  # even extents, the volume spread over its logarithm; T from half of L to four times L
        v = math.exp(rng.uniform(math.log(least), math.log(most)))
        r = math.exp(rng.uniform(math.log(0.5), math.log(4.0)))
        L = max(4, 2 * round((v / r) ** 0.25 / 2))
        T = max(4, 2 * round(v / L ** 3 / 2))
        if least <= T * L ** 3 <= most and T <= 128:
            break
    V = T * L ** 3
    if kind == "hop":
        prec, link = rng.choice([("f64", 18), ("f32", 18), ("f32", 12), ("f16", 12), ("f16", 8)])
        nrhs = rng.choice([1, 1, 1, 2, 3]) if 3 * V <= most else 1
        return dict(kind=kind, T=T, L=L, prec=prec, link=link, parity=rng.randrange(2), nrhs=nrhs)
    if kind == "dirac":
        nrhs = rng.choice([1, 1, 2, 3]) if 3 * V <= most else 1
        return dict(kind=kind, T=T, L=L, nrhs=nrhs, flavour=rng.choice([1, -1]), dagger=rng.random() < 0.5)
    if kind == "fields":
        return dict(kind=kind, T=T, L=L, prec=rng.choice(["f64", "f32", "f16"]), nrhs=rng.choice([1, 2, 3]))
    if kind == "solve":
        if rng.random() < 0.5:
            return dict(kind=kind, T=T, L=L, prec="f32", link=rng.choice([12, 18]), delta=1e-5, upd="f64")
        return dict(kind=kind, T=T, L=L, prec="f16", link=rng.choice([12, 8]), delta=0.1, upd="f64")
    return dict(kind=kind, T=T, L=L)


# ------------------------------------------------------------------- inputs ---
def _params(c):
    """eps, kappa, mu of the package's workloads at this size."""
    return (0.6, 0.1615, 0.003) if c["T"] * c["L"] ** 3 > 16 ** 3 * 32 else (0.5, 0.1632, 0.004)


def _gen(seed, what):
    return torch.Generator(device="cuda").manual_seed(seed * 8 + what)


def _normal(shape, g):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)


def _gauge(c, seed):
    """Random links near exp(i eps H) made exactly unitary, (T, L, L, L, 4, 3, 3) complex128."""
    T, L = c["T"], c["L"]
    g = _gen(seed, 0)
    eps = _params(c)[0]
    U = torch.empty((T, L * L * L * 4, 3, 3), device="cuda", dtype=torch.complex128)
    for t in range(0, T, 16):  # by time slices: bounded temporaries
        n = min(16, T - t)
        h = torch.randn((n, L * L * L * 4, 8), generator=g, device="cuda").double() * (0.5 * eps)
        d = h[..., 7] / math.sqrt(3.0)
        off = [torch.complex(h[..., 2 * k], h[..., 2 * k + 1]) for k in range(3)]  # entries 01, 02, 12
        diag = [h[..., 6] + d, d - h[..., 6], -2.0 * d]
        H = [[diag[0] + 0j, off[0].conj(), off[1].conj()], [off[0], diag[1] + 0j, off[2].conj()]]
        rows = []
        for a in range(2):  # rows 0 and 1 of 1 + i H - H^2 / 2, then Gram-Schmidt
            full = [[diag[0] + 0j, off[0].conj(), off[1].conj()], [off[0], diag[1] + 0j, off[2].conj()],
                    [off[1], off[2], diag[2] + 0j]]
            rows.append([1j * H[a][b] - 0.5 * sum(H[a][k] * full[k][b] for k in range(3)) + (1.0 if a == b else 0.0)
                         for b in range(3)])
        nrm = torch.rsqrt(sum(x.abs() ** 2 for x in rows[0]))
        r0 = [x * nrm for x in rows[0]]
        p = sum(x.conj() * y for x, y in zip(r0, rows[1]))
        r1 = [y - p * x for x, y in zip(r0, rows[1])]
        nrm = torch.rsqrt(sum(x.abs() ** 2 for x in r1))
        r1 = [x * nrm for x in r1]
        r2 = [(r0[1] * r1[2] - r0[2] * r1[1]).conj(), (r0[2] * r1[0] - r0[0] * r1[2]).conj(),
              (r0[0] * r1[1] - r0[1] * r1[0]).conj()]
        for a, r in enumerate((r0, r1, r2)):
            for b in range(3):
                U[t:t + n, :, a, b] = r[b]
    return U.view(T, L, L, L, 4, 3, 3)


def _spinor(shape, g):
    return torch.view_as_complex(_normal(tuple(shape) + (2,), g) * math.sqrt(0.5))


def _canonical(c, seed):
    """The canonical input fields of a case (complex128)."""
    T, L = c["T"], c["L"]
    n = c.get("nrhs", 1)
    if c["kind"] in ("hop", "fields", "normal"):
        return _spinor((n, T * L ** 3 // 2, 4, 3), _gen(seed, 1))
    if c["kind"] == "contract":
        t = torch.arange(T, device="cuda", dtype=torch.float64)
        decay = torch.exp(-0.3 * torch.minimum(t, T - t)).view(1, T, 1, 1, 1, 1, 1)
        return _spinor((12, T, L, L, L, 4, 3), _gen(seed, 1)) * decay
    if c["kind"] == "points":
        b = torch.zeros((12, T, L, L, L, 4, 3), device="cuda", dtype=torch.complex128)
        for j in range(12):
            b[j, 0, 0, 0, 0, j // 3, j % 3] = 1.0
        return b
    return _spinor((n, T, L, L, L, 4, 3), _gen(seed, 1))


def _correlator_matrices():
    """X = Gamma gamma5 of C_PP, C_PA (Gamma = gamma0 gamma5) and C_PV (Gamma = gamma0)."""
    one = np.eye(4, dtype=np.complex128)
    g0 = np.zeros((4, 4), dtype=np.complex128)
    g0[0, 2] = g0[1, 3] = g0[2, 0] = g0[3, 1] = -1.0
    return torch.from_numpy(np.stack([one, g0, g0 @ np.diag([1.0, 1.0, -1.0, -1.0])])).to("cuda")


def prepare(case, seed):
    c = dict(case)
    T, L, n = c["T"], c["L"], c.get("nrhs", 1)
    _, kappa, mu = _params(c)
    s = {"case": c, "lat": tm.Lattice(T, L, kappa, mu)}
    lat = s["lat"]
    src = _canonical(c, seed)
    if c["kind"] not in ("fields", "contract"):
        lat.set_gauge(_gauge(c, seed))
    if c["kind"] == "hop":
        p = PREC[c["prec"]]
        s["in"] = torch.empty((n, lat.half_field_bytes(p)), device="cuda", dtype=torch.uint8)
        s["out"] = torch.zeros_like(s["in"])
        lat.pack_half(p, s["in"], src, nrhs=n)
        # the gauge copy of this storage form, which a program builds once per gauge field
        lat.apply_hopping_eo(c["parity"], s["out"], s["in"], prec=p, link=c["link"], nrhs=n)
    elif c["kind"] == "fields":
        s["in"] = src
        s["half"] = torch.empty((n, lat.half_field_bytes(PREC[c["prec"]])), device="cuda", dtype=torch.uint8)
        s["out"] = torch.zeros_like(src)
    elif c["kind"] == "normal":
        s["in"] = torch.empty(lat.half_field_bytes(F64), device="cuda", dtype=torch.uint8)
        s["out"] = torch.zeros_like(s["in"])
        lat.pack_half(F64, s["in"], src)
    elif c["kind"] == "contract":
        s["in"] = src
        s["out"] = torch.zeros((T, 12, 12), device="cuda", dtype=torch.complex128)
        s["X"] = _correlator_matrices()
    else:
        s["in"] = src
        s["out"] = torch.zeros_like(src)
    torch.cuda.synchronize()
    return s


def _typed(buf, prec, h):
    """Stacked half fields as numbers: FP64 / FP32 blocks, or the halves and the norms of FP16 storage."""
    if prec == "f16":
        return buf[:, :48 * h].view(torch.float16), buf[:, 48 * h:].view(torch.float32)
    return buf.view(torch.float64 if prec == "f64" else torch.float32)


def run(state):
    c, lat, x, out = state["case"], state["lat"], state["in"], state["out"]
    kind = c["kind"]
    if kind == "hop":
        lat.apply_hopping_eo(c["parity"], out, x, prec=PREC[c["prec"]], link=c["link"], nrhs=c["nrhs"])
        return _typed(out, c["prec"], lat.h)
    if kind == "dirac":
        lat.apply_D(out, x, flavour=c["flavour"], dagger=c["dagger"], nrhs=c["nrhs"])
        return out
    if kind == "fields":
        p = PREC[c["prec"]]
        lat.pack_half(p, state["half"], x, nrhs=c["nrhs"])
        lat.unpack_half(p, out, state["half"], nrhs=c["nrhs"])
        return _typed(state["half"], c["prec"], lat.h), out
    if kind == "solve":
        lat.solve_cg(out, x, tol=1e-10, mode=tm.CG_RELIABLE, sloppy_prec=PREC[c["prec"]], sloppy_link=c["link"],
                     delta=c["delta"], update_prec=PREC[c["upd"]])
        return out
    if kind == "normal":
        lat.solve_normal(out, x, tol=1e-10)
        return out.view(torch.float64)
    if kind == "points":
        tm.solve_cg_batch([(lat, lat.mu, out[j], x[j], -1) for j in range(12)], tol=1e-10,
                          sloppy_prec=PREC[c["prec"]], sloppy_link=c["link"], delta=c["delta"])
        return out
    lat.meson_contract(x, out=out)
    return out, tm.correlator(lat, out, state["X"])


# --------------------------------------------------------------------- work ---
def work(case):
    c = case
    V = c["T"] * c["L"] ** 3
    h = V // 2
    n = c.get("nrhs", 1)
    site = {"f64": 192, "f32": 96, "f16": 52}
    real = {"f64": 8, "f32": 4, "f16": 2}
    kind = c["kind"]
    if kind == "hop":  # fields in and out, the 8 links of an output site (each link used once)
        return {"bytes": h * (2 * n * site[c["prec"]] + 8 * c["link"] * real[c["prec"]]), "flops": 1320 * h * n}
    if kind == "dirac":  # fields in and out, every link once (18 reals)
        return {"bytes": V * (2 * 192 * n + 4 * 144), "flops": 1392 * V * n}
    if kind == "fields":
        return {"bytes": n * h * 2 * (192 + site[c["prec"]]), "flops": 0}
    if kind in ("solve", "points", "normal"):
        # one iteration: 4 hopping terms and the vector updates, at the iterations these systems take
        n, p, link, iters = (12, c["prec"], c["link"], 88) if kind == "points" else (
            (1, c["prec"], c["link"], 88) if kind == "solve" else (1, "f64", 18, 88))
        links = 4 * 8 * link * real[p] * h
        return {"bytes": iters * (links + n * 14 * site[p] * h), "flops": iters * n * 4 * 1392 * h}
    return {"bytes": 12 * 192 * V, "flops": 78 * 12 * 8 * V}  # contract


# -------------------------------------------------------------------- exact ---
# gamma_mu psi (chiral basis): component s is phase[s] * psi[partner[s]]
_GAMMA = [((2, 3, 0, 1), (-1, -1, -1, -1)),      # t
          ((3, 2, 1, 0), (-1j, -1j, 1j, 1j)),    # x
          ((3, 2, 1, 0), (-1, 1, 1, -1)),        # y
          ((2, 3, 0, 1), (-1j, 1j, 1j, -1j))]    # z
_AXIS = (-6, -3, -4, -5)  # t, x, y, z of (..., t, z, y, x, spin, colour)


def _mul(U, v):
    """U v, entry by entry (U: (..., 3, 3), v: (..., spin, 3))."""
    return torch.stack([sum(U[..., a, b].unsqueeze(-1) * v[..., b] for b in range(3)) for a in range(3)], -1)


def _hop(U, psi):
    """sum_mu U (1 + gamma) psi(x + mu) + U(x - mu)^dag (1 - gamma) psi(x - mu); -1 across the time boundary."""
    out = torch.zeros_like(psi)
    for mu in range(4):
        partner, phase = _GAMMA[mu]
        ph = torch.tensor(phase, device=psi.device, dtype=psi.dtype).view(4, 1)
        g = psi[..., list(partner), :] * ph
        u = U[..., mu, :, :]
        f = torch.roll(psi + g, -1, _AXIS[mu])
        b = _mul(u.conj().transpose(-1, -2), psi - g)
        if mu == 0:
            f[..., -1, :, :, :, :, :] *= -1
            b[..., -1, :, :, :, :, :] *= -1
        out += _mul(u, f)
        out += torch.roll(b, 1, _AXIS[mu])
    return out


def _g5(psi):
    return psi * torch.tensor([1.0, 1.0, -1.0, -1.0], device=psi.device).view(4, 1)


def _M(U, psi, kappa, mut):
    return psi + 1j * mut * _g5(psi) - kappa * _hop(U, psi)


def _mask(c, parity):
    T, L = c["T"], c["L"]
    r = lambda n: torch.arange(n, device="cuda")  # noqa: E731
    return (r(T).view(T, 1, 1, 1) + r(L).view(L, 1, 1) + r(L).view(L, 1) + r(L)) % 2 == parity


def _blocks(v, prec):
    """(n, h, 4, 3) complex in the block order of a storage form, as real numbers; FP16: halves and norms."""
    n, h = v.shape[:2]
    x = torch.view_as_real(v.reshape(n, h, 12))
    if prec == "f64":
        return x.permute(0, 2, 1, 3).contiguous()
    if prec == "f32":
        return x.reshape(n, h, 6, 2, 2).permute(0, 2, 1, 3, 4).contiguous()
    m = x.abs().amax((2, 3))
    y = x / m.view(n, h, 1, 1)
    return y.reshape(n, h, 3, 4, 2).permute(0, 2, 1, 3, 4).contiguous().view(n, -1), m


def _stored(v, prec):
    """What a storage form holds of the FP64 half fields v."""
    if prec == "f64":
        return v
    x = torch.view_as_real(v)
    if prec == "f32":
        return torch.view_as_complex(x.float().double())
    m = x.abs().amax((2, 3, 4), keepdim=True).float()
    return torch.view_as_complex((x.float() / m).half().double() * m.double())


def _cg(apply, b):
    """Conjugate gradients in complex128 for each field of b (first axis), far below the solver's tolerance."""
    dims = tuple(range(1, b.dim()))
    dot = lambda u, v: (u.conj() * v).real.sum(dims, keepdim=True)  # noqa: E731
    x, r, p = torch.zeros_like(b), b.clone(), b.clone()
    rr = dot(r, r)
    stop = rr * 1e-28
    for _ in range(1000):
        a = apply(p)
        al = rr / dot(p, a)
        x += al * p
        r -= al * a
        new = dot(r, r)
        if bool((new < stop).all()):
            break
        p = r + (new / rr) * p
        rr = new
    return x


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    _, kappa, mu = _params(c)
    mut = 2 * kappa * mu
    src = _canonical(c, seed)
    V = c["T"] * c["L"] ** 3
    if kind == "fields":
        kept = _stored(src, c["prec"])
        return _blocks(src, c["prec"]), kept
    if kind == "contract":
        x = src.reshape(12, c["T"], -1)
        A = torch.einsum("jts,kts->tjk", x.conj(), x)
        C = torch.einsum("tacbc,gba->gt", A.view(c["T"], 4, 3, 4, 3), _correlator_matrices())
        return A, C
    U = _gauge(c, seed)
    if kind == "hop":
        full = torch.zeros((c["nrhs"],) + tuple(U.shape[:4]) + (4, 3), device="cuda", dtype=torch.complex128)
        full[:, _mask(c, 1 - c["parity"])] = _stored(src, c["prec"])
        return _blocks(torch.stack([_hop(U, f)[_mask(c, c["parity"])] for f in full]), c["prec"])
    if kind == "dirac":
        m = c["flavour"] * mut
        one = lambda v: _g5(_M(U, _g5(v), kappa, -m)) if c["dagger"] else _M(U, v, kappa, m)  # noqa: E731
        return torch.stack([one(v) for v in src])
    if kind == "points" or V > 16 ** 3 * 32:
        return None
    if kind == "solve":
        Md = lambda v: _g5(_M(U, _g5(v), kappa, -mut))  # noqa: E731
        return _cg(lambda v: Md(_M(U, v, kappa, mut)), Md(src))
    # normal: Qhat^+ Qhat^- X = phi on the odd sites, Qhat^f = gamma5 [(1 + i f mut g5) - kappa^2 H (1 + i f mut g5)^-1 H]
    even, odd = _mask(c, 0).view(c["T"], c["L"], c["L"], c["L"], 1, 1), _mask(c, 1)
    site = lambda v, m: v + 1j * m * _g5(v)  # noqa: E731
    Q = lambda v, f: _g5(site(v, f * mut) - kappa ** 2 * (  # noqa: E731
        _hop(U, even * site(_hop(U, v), -f * mut) / (1 + mut * mut)) * ~even))
    phi = torch.zeros((1,) + tuple(U.shape[:4]) + (4, 3), device="cuda", dtype=torch.complex128)
    phi[:, odd] = src
    return _blocks(_cg(lambda v: Q(Q(v, -1), 1), phi)[:, odd], "f64")
