"""Measured cases: the calls that a lattice program makes of this library, over the sizes they have in use.

A case is a dict of plain values.  ``kind`` names the call:

* ``hop``    the Wilson operator on one field: ``dslash_apply`` / ``dslash_apply_dagger`` on full
             fields, ``dslash_eo_apply`` on half fields (``full`` False) with or without the axpy term;
* ``mrhs``   the same on several right-hand sides of one gauge field (a propagator's 12 sources);
* ``pack``   canonical array -> device field -> canonical array (``wd.pack``, ``wd.unpack``);
* ``blas``   the vector work between operator applications: axpby, inner product, norm, conversion;
* ``cg``     ``cg_solve`` on the even-odd normal equations, mixed precision;
* ``batch``  ``cg_solve_batch`` in graph mode: the request groups behind the serving queue.

Launch shapes are the library's own defaults (no autotuning run), as for a program that just calls it.
"""
import torch

import paper_1901_07294_gb300 as wd

PREC = {"f64": wd.F64, "f32": wd.F32, "f16": wd.F16, "bf16": wd.BF16, "df": wd.DF}
FIELD_REAL = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2, "df": 8}   # bytes of a stored real
SCALE = {"f64": 0, "f32": 0, "f16": 4, "bf16": 4, "df": 0}        # bytes of the per-site scale
LINK_EPS = 0.2   # smoothed links near the unit matrix, as in the tests and the benchmark

_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = wd.Context(0)
    return _ctx


# ---- the cases -------------------------------------------------------------------------------

def _hop(name, dims, prec, recon, full, dagger=False, with_x=False, nrhs=1):
    return {"name": name, "kind": "hop" if nrhs == 1 else "mrhs", "lx": dims[0], "ly": dims[1], "lz": dims[2],
            "lt": dims[3], "prec": prec, "recon": recon, "full": full, "dagger": dagger, "with_x": with_x, "nrhs": nrhs}


def listed():
    return [
        # the smallest lattice of the parity tests: one call is launch and latency
        _hop("full_f32_8", (8, 8, 8, 8), "f32", 18, True),
        # the operator on an ordinary lattice in the smallest storage (compressed links), Eq. (1)'s own sign convention
        _hop("full_bf16_r12_16x32", (16, 16, 16, 32), "bf16", 12, True, dagger=True),
        # the benchmark's headline: the single-precision operator on 32^4
        _hop("full_f32_32", (32, 32, 32, 32), "f32", 18, True),
        # one of the four hops of a mixed-precision CG iteration on the solver lattice
        _hop("eo_f16_24x48", (24, 24, 24, 48), "f16", 18, False, dagger=True, with_x=True),
        # the same hop of the double-precision solve and of its convergence checks
        _hop("eo_f64_24x48", (24, 24, 24, 48), "f64", 18, False, with_x=True),
        # the same hop of the double-word reliable updates
        _hop("eo_df_24x48", (24, 24, 24, 48), "df", 18, False, with_x=True),
        # a propagator's 12 sources on one gauge field
        _hop("mrhs12_eo_f32_32", (32, 32, 32, 32), "f32", 18, False, nrhs=12),
        # a few sources on a small lattice of odd proportions
        _hop("mrhs5_full_f16_ragged", (12, 14, 10, 18), "f16", 18, True, nrhs=5),
        # a field into the library and back, single precision on both sides
        {"name": "pack_f32_32", "kind": "pack", "lx": 32, "ly": 32, "lz": 32, "lt": 32, "prec": "f32", "canon": "f32",
         "half": False},
        # the vector work of one mixed-precision iteration on the solver lattice
        {"name": "blas_f16_24x48", "kind": "blas", "lx": 24, "ly": 24, "lz": 24, "lt": 48, "prec": "f16", "half": True},
        # the mixed-precision solve on the solver lattice, to the tightest tolerance of the serving mix
        {"name": "cg_f16_24x48", "kind": "cg", "lx": 24, "ly": 24, "lz": 24, "lt": 48, "prec": "f16", "outer": "df",
         "mass": 0.1, "tol": 1e-12, "graph": True},
        # a batch of uneven masses on one gauge field
        {"name": "batch6_f16_16", "kind": "batch", "lx": 16, "ly": 16, "lz": 16, "lt": 16, "prec": "f16", "outer": "df",
         "tol": 1e-12, "n": 6},
    ]


def _extents(rng, most, least=4):
    """Even extents, spread over their logarithm, of at most `most` sites."""
    while True:
        d = [2 * max(least // 2, round(0.5 * least * (32 / least) ** rng.random())) for _ in range(3)]
        d.append(2 * max(least // 2, round(0.5 * least * (48 / least) ** rng.random())))
        if d[0] * d[1] * d[2] * d[3] <= most:
            return dict(zip(("lx", "ly", "lz", "lt"), d))


def draw(rng):
    kind = rng.choice(["hop", "hop", "hop", "mrhs", "mrhs", "pack", "blas", "cg", "batch"])
    if kind == "hop":
        prec = rng.choice(["f64", "f32", "f32", "f16", "f16", "bf16", "df"])
        c = _extents(rng, 663552 if prec in ("f64", "df") else 1048576)
        full = rng.random() < 0.5
        return {"kind": kind, **c, "prec": prec, "recon": rng.choice([18, 18, 12]), "full": full,
                "dagger": rng.random() < 0.5, "with_x": not full and rng.random() < 0.5, "nrhs": 1}
    if kind == "mrhs":
        full = rng.random() < 0.5
        return {"kind": kind, **_extents(rng, 524288), "prec": rng.choice(["f32", "f32", "f16", "bf16"]),
                "recon": rng.choice([18, 18, 12]), "full": full, "dagger": rng.random() < 0.5,
                "with_x": not full and rng.random() < 0.5, "nrhs": rng.randint(2, 13)}
    if kind == "pack":
        return {"kind": kind, **_extents(rng, 1048576), "prec": rng.choice(["f64", "f32", "f16", "bf16"]),
                "canon": rng.choice(["f64", "f32"]), "half": rng.random() < 0.3}
    if kind == "blas":
        return {"kind": kind, **_extents(rng, 1048576, 8), "prec": rng.choice(["f64", "f32", "f16", "bf16"]),
                "half": rng.random() < 0.6}
    prec = rng.choice(["f32", "f16", "f16", "bf16"])
    c = {"kind": kind, **_extents(rng, 131072, 8), "prec": prec, "outer": rng.choice(["df", "f64"]), "tol": 1e-12}
    if kind == "cg":
        return {**c, "mass": round(rng.uniform(0.05, 0.5), 3), "graph": rng.random() < 0.5}
    return {**c, "n": rng.randint(2, 8)}


# ---- inputs ----------------------------------------------------------------------------------

def _dims(case):
    return (case["lx"], case["ly"], case["lz"], case["lt"])


def _volume(case):
    return case["lx"] * case["ly"] * case["lz"] * case["lt"]


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _links(volume, seed):
    """Random SU(3) matrices near the unit matrix, (V, 4, 3, 3): the rows of 1 + i eps H
    orthonormalised, the third one closing the determinant."""
    a = torch.randn(volume, 4, 3, 3, dtype=torch.complex128, device="cuda", generator=_generator(2 * seed))
    h = a + a.mH   # entries of mean square 2, scaled to 1 below
    del a
    h.mul_(1j * LINK_EPS / 2 ** 0.5)
    h.diagonal(dim1=-2, dim2=-1).add_(1.0)
    r0 = h[..., 0, :] / torch.linalg.vector_norm(h[..., 0, :], dim=-1, keepdim=True)
    r1 = h[..., 1, :] - r0 * (r0.conj() * h[..., 1, :]).sum(-1, keepdim=True)
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    h[..., 0, :] = r0
    h[..., 1, :] = r1
    h[..., 2, :] = torch.linalg.cross(r0, r1).conj()
    return h


def _spinors(volume, n, seed, dtype=torch.float64):
    """n Gaussian sources, (n, V, 24) reals."""
    return torch.randn(n, volume, 24, dtype=dtype, device="cuda", generator=_generator(2 * seed + 1))


def _sites(case):
    """(wd_sites value, number of half fields) of the case's fields."""
    half = case["half"] if "half" in case else not case.get("full", False)
    return (wd.SITES_EVEN, 1) if half else (wd.SITES_FULL, 2)


def _values(buf, case, prec, nhalf, n=1):
    """The stored numbers of a device field, by type: views of its planes and of its per-site scales."""
    vh = _volume(case) // 2
    main = 24 * FIELD_REAL[prec] * vh
    kind = {"f64": torch.float64, "f32": torch.float32, "df": torch.float32, "f16": torch.float16,
            "bf16": torch.bfloat16}[prec]
    rows = buf.view(n * nhalf, main + SCALE[prec] * vh)
    out = [rows[:, :main].view(kind)]
    if SCALE[prec]:
        out.append(rows[:, main:].view(torch.float32))
    return out


def _pack(case, prec, sites, aos):
    """The n canonical spinors of aos, one after another, in one device buffer."""
    one = wd.field_bytes(_dims(case), sites, PREC[prec])
    buf = torch.empty(aos.shape[0] * one, dtype=torch.uint8, device="cuda")
    for k in range(aos.shape[0]):
        wd.pack(_context(), _dims(case), sites, PREC[prec], aos[k], buf[k * one:(k + 1) * one])
    return buf


def _gauge(case, seed):
    links = _links(_volume(case), seed)
    torch.cuda.synchronize()   # the gauge is built on a stream of its own
    return wd.Gauge(_context(), _dims(case), links)


def _masses(n, seed):
    r = torch.rand(n, dtype=torch.float64, generator=torch.Generator().manual_seed(int(seed)))
    return [0.05 + 0.45 * float(v) for v in r]


def prepare(case, seed):
    ctx, dims, v = _context(), _dims(case), _volume(case)
    kind, prec = case["kind"], case["prec"]
    if kind in ("hop", "mrhs"):
        n = case["nrhs"]
        g = _gauge(case, seed)
        g.prepare(PREC[prec], case["recon"])
        in_sites, nhalf = (wd.SITES_FULL, 2) if case["full"] else (wd.SITES_ODD, 1)
        psi = _spinors(v, n, seed)
        s = {"kind": kind, "case": case, "gauge": g, "inp": _pack(case, prec, in_sites, psi), "x": None}
        if case["with_x"]:
            s["x"] = _pack(case, prec, wd.SITES_EVEN, psi)
        s["out"] = torch.zeros_like(s["inp"])
        s["values"] = _values(s["out"], case, prec, nhalf, n)
        return s
    if kind == "pack":
        sites, nhalf = _sites(case)
        dtype = torch.float32 if case["canon"] == "f32" else torch.float64
        s = {"kind": kind, "case": case, "sites": sites, "aos": _spinors(v, 1, seed, dtype)[0]}
        s["field"] = torch.zeros(wd.field_bytes(dims, sites, PREC[prec]), dtype=torch.uint8, device="cuda")
        s["back"] = torch.zeros_like(s["aos"])
        s["values"] = _values(s["field"], case, prec, nhalf)
        return s
    if kind == "blas":
        sites, nhalf = _sites(case)
        xy = _spinors(v, 2, seed)
        s = {"kind": kind, "case": case, "sites": sites, "x": _pack(case, prec, sites, xy[:1]),
             "y": _pack(case, prec, sites, xy[1:]), "res": torch.zeros(3, dtype=torch.float64, device="cuda")}
        s["z"] = torch.zeros(wd.field_bytes(dims, sites, wd.F32), dtype=torch.uint8, device="cuda")
        s["dot"], s["norm"] = s["res"][:2], s["res"][2:]
        s["values"] = [s["res"], *_values(s["y"], case, prec, nhalf), *_values(s["z"], case, "f32", nhalf)]
        return s
    g = _gauge(case, seed)
    for p in {prec, case["outer"], "f64"}:
        g.prepare(PREC[p], 18)
    n = case.get("n", 1)
    b = _pack(case, "f64", wd.SITES_EVEN, _spinors(v, n, seed)).view(n, -1)
    x = torch.zeros_like(b)
    s = {"kind": kind, "case": case, "gauge": g, "b": b, "x": x, "values": x.view(torch.float64)}
    if kind == "batch":
        s["problems"] = [{"gauge": g, "mass": m, "tol": case["tol"], "x": x[k], "b": b[k], "inner_prec": PREC[prec],
                          "outer_prec": PREC[case["outer"]]} for k, m in enumerate(_masses(n, seed))]
    return s


def run(s):
    c, ctx = s["case"], _ctx
    if s["kind"] in ("hop", "mrhs"):
        if c["full"]:
            apply = wd.dslash_apply_dagger if c["dagger"] else wd.dslash_apply
            apply(ctx, s["gauge"], s["out"], s["inp"], 0.1, nrhs=c["nrhs"], prec=PREC[c["prec"]], recon=c["recon"])
        elif s["x"] is None:   # the hopping term alone (H_oe, H_eo)
            wd.dslash_eo_apply(ctx, s["gauge"], s["out"], s["inp"], None, wd.EVEN, 0.0, 1.0, dagger=c["dagger"],
                               nrhs=c["nrhs"], prec=PREC[c["prec"]], recon=c["recon"])
        else:                  # the second hop of the Schur complement
            wd.dslash_eo_apply(ctx, s["gauge"], s["out"], s["inp"], s["x"], wd.EVEN, 4.1, -1.0 / 16.4,
                               dagger=c["dagger"], nrhs=c["nrhs"], prec=PREC[c["prec"]], recon=c["recon"])
        return s["values"]
    if s["kind"] == "pack":
        wd.pack(ctx, _dims(c), s["sites"], PREC[c["prec"]], s["aos"], s["field"])
        wd.unpack(ctx, _dims(c), s["sites"], PREC[c["prec"]], s["field"], s["back"])
        return [*s["values"], s["back"]]
    if s["kind"] == "blas":
        d, sites, p = _dims(c), s["sites"], PREC[c["prec"]]
        wd.axpby(ctx, d, sites, p, 0.75, s["x"], 0.5, s["y"])
        wd.dot(ctx, d, sites, p, s["x"], s["y"], s["dot"])
        wd.norm2(ctx, d, sites, p, s["y"], s["norm"])
        wd.convert(ctx, d, sites, wd.F32, s["z"], p, s["y"])
        return s["values"]
    if s["kind"] == "cg":
        wd.cg_solve(ctx, s["gauge"], c["mass"], s["x"], s["b"], tol=c["tol"], inner_prec=PREC[c["prec"]],
                    use_graph=c["graph"], outer_prec=PREC[c["outer"]])
        return s["values"]
    wd.cg_solve_batch(ctx, s["problems"], mode=wd.BATCH_GRAPH)
    return s["values"]


# ---- work ------------------------------------------------------------------------------------

def work(case):
    v, kind, prec = _volume(case), case["kind"], case["prec"]
    field = 24 * FIELD_REAL[prec] + SCALE[prec]   # bytes of one site's spinor
    if kind in ("hop", "mrhs"):
        link = case["recon"] * {"f64": 8, "f32": 4, "df": 8}.get(prec, 2)
        sites = v if case["full"] else v // 2
        fields = 3 if case["with_x"] else 2
        return {"bytes": case["nrhs"] * sites * fields * field + 4 * v * link, "flops": case["nrhs"] * sites * 1320}
    sites = v // 2 * (_sites(case)[1] if kind in ("pack", "blas") else 1)
    if kind == "pack":
        canon = 96 if case["canon"] == "f32" else 192
        return {"bytes": 2 * sites * (canon + field), "flops": 0}
    if kind == "blas":   # axpby 3 fields, dot 2, norm 1, conversion 1 and an FP32 one
        return {"bytes": sites * (7 * field + 96), "flops": sites * (72 + 96 + 48)}
    # a solve: its source and links in, its solution out, and the operator in the storage of the iteration, which
    # cannot converge in fewer than about 60 applications of four hops (masses 0.05 to 0.5, these tolerances)
    n = case.get("n", 1)
    hop = 2 * sites * field * n + 4 * v * 18 * {"f32": 4}.get(prec, 2)
    return {"bytes": 2 * 192 * sites * n + 4 * 60 * hop, "flops": n * 60 * 4 * 1320 * sites}


# ---- the same in 64 bits, by plain torch -----------------------------------------------------

# gamma_mu in the chiral basis: row r has one entry, (column, value)
_GAMMA = [[(3, 1j), (2, 1j), (1, -1j), (0, -1j)], [(3, -1), (2, 1), (1, 1), (0, -1)],
          [(2, 1j), (3, -1j), (0, -1j), (1, 1j)], [(2, 1), (3, 1), (0, 1), (1, 1)]]


def _project(psi, mu, sign):
    """(1 + sign gamma_mu) psi."""
    cols = [c for c, _ in _GAMMA[mu]]
    vals = torch.tensor([complex(f) for _, f in _GAMMA[mu]], dtype=torch.complex128, device=psi.device)
    return psi + sign * vals[:, None] * psi[..., cols, :]


def _times(u, psi, adjoint):
    """U psi or U^dagger psi on the colour index, site by site."""
    out = None
    for b in range(3):
        col = u[..., b, :].conj() if adjoint else u[..., :, b]
        t = col[..., None, :] * psi[..., :, b, None]
        out = t if out is None else out.add_(t)
    return out


def _hopping(dims, u, psi, dagger):
    """H psi on the whole lattice (gamma5 H gamma5 with dagger); psi (T, Z, Y, X, 4, 3)."""
    sign = 1 if dagger else -1
    out = torch.zeros_like(psi)
    for mu in range(4):
        axis = 3 - mu
        um = u[..., mu, :, :]
        out += _project(_times(um, torch.roll(psi, -1, axis), False), mu, sign)
        out += _project(torch.roll(_times(um, psi, True), 1, axis), mu, -sign)
    return out


def _lattice(case, reals):
    lx, ly, lz, lt = _dims(case)
    return torch.view_as_complex(reals.double().reshape(lt, lz, ly, lx, 4, 3, 2).contiguous())


def _odd(case):
    """Sites of odd x + y + z + t, in lexicographic order."""
    lx, ly, lz, lt = _dims(case)
    r = [torch.arange(n, device="cuda") for n in (lt, lz, ly, lx)]
    return ((r[0][:, None, None, None] + r[1][:, None, None] + r[2][:, None] + r[3]) & 1).reshape(-1).bool()


def _half_fields(case, psi, which):
    """(half fields, V/2, 24) reals of the named parities, sites in lexicographic order."""
    rows = torch.view_as_real(psi.contiguous()).reshape(-1, 24)
    odd = _odd(case)
    return torch.stack([rows[odd] if p else rows[~odd] for p in which])


def _stored(halves, prec):
    """The numbers a field of precision prec holds for these half fields: as _values lays them out."""
    n, vh, _ = halves.shape
    if prec == "df":
        hi = halves.float()
        lo = (halves - hi.double()).float()
        halves = torch.stack([hi, lo], -1).reshape(n, vh, 48).double()
        per = 4
    else:
        per = 16 // FIELD_REAL[prec]
    scale = None
    if SCALE[prec]:
        scale = halves.abs().amax(-1, keepdim=True)
        halves = halves / scale
    rows = halves.reshape(n, vh, -1, per).permute(0, 2, 1, 3).reshape(n, -1)
    return [rows] if scale is None else [rows, scale.reshape(n, vh)]


def _rows(parts):
    return [torch.cat(p) for p in zip(*parts)]


def _normal(dims, u, odd, mass, v):
    """Mhat^dagger Mhat v for v on the even sites (zero elsewhere)."""
    a = mass + 4.0
    for dagger in (False, True):
        t = _hopping(dims, u, v, dagger) * odd
        v = a * v - (_hopping(dims, u, t, dagger) * ~odd) / (4.0 * a)
    return v


def _solve(dims, u, odd, mass, b):
    """Conjugate gradient in 64 bits, down to the rounding of the residual."""
    dot = lambda p, q: torch.vdot(p.reshape(-1), q.reshape(-1)).real   # noqa: E731
    x, r = torch.zeros_like(b), b.clone()
    p, r2 = r.clone(), dot(r, r)
    stop = 1e-28 * float(r2)
    for _ in range(400):
        ap = _normal(dims, u, odd, mass, p)
        alpha = r2 / dot(p, ap)
        x += alpha * p
        r -= alpha * ap
        new = dot(r, r)
        if float(new) <= stop:
            break
        p = r + (new / r2) * p
        r2 = new
    return x


def exact(case, seed):
    dims, v = _dims(case), _volume(case)
    kind, prec = case["kind"], case["prec"]
    if kind == "pack":
        dtype = torch.float32 if case["canon"] == "f32" else torch.float64
        aos = _spinors(v, 1, seed, dtype)[0].double()
        half = _sites(case)[1] == 1
        back = aos.clone()
        if half:
            back[_odd(case)] = 0.0
        return [*_stored(_half_fields(case, _lattice(case, aos), (0,) if half else (0, 1)), prec), back]
    if kind == "blas":
        which = (0,) if _sites(case)[1] == 1 else (0, 1)
        x, y = (_half_fields(case, _lattice(case, r), which) for r in _spinors(v, 2, seed))
        y = 0.75 * x + 0.5 * y
        cx, cy = (torch.view_as_complex(r.reshape(-1, 2)) for r in (x, y))
        d = torch.vdot(cx, cy)
        res = torch.stack([d.real, d.imag, torch.vdot(cy, cy).real])
        if prec != "f64":   # sums over stored, rounded values: no number of their own in 64 bits
            res = None
        return [res, *_stored(y, prec), *_stored(y, "f32")]
    lx, ly, lz, lt = dims
    u = _links(v, seed).reshape(lt, lz, ly, lx, 4, 3, 3)
    odd = _odd(case).reshape(lt, lz, ly, lx, 1, 1)
    if kind in ("hop", "mrhs"):
        parts = []
        for k, r in enumerate(_spinors(v, case["nrhs"], seed)):
            psi = _lattice(case, r)
            if case["full"]:
                out = 4.1 * psi - 0.5 * _hopping(dims, u, psi, case["dagger"])
            else:
                out = _hopping(dims, u, psi * odd, case["dagger"])
                if case["with_x"]:
                    out = 4.1 * psi - out / 16.4
            parts.append(_stored(_half_fields(case, out, (0, 1) if case["full"] else (0,)), prec))
        return _rows(parts)
    masses = [case["mass"]] if kind == "cg" else _masses(case["n"], seed)
    rows = []
    for m, r in zip(masses, _spinors(v, len(masses), seed)):
        x = _solve(dims, u, odd, m, _lattice(case, r) * ~odd)
        rows.append(_stored(_half_fields(case, x, (0,)), "f64")[0])
    return torch.cat(rows)
