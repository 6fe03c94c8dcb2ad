"""Performance cases: the calls a lattice program makes into the library, over the range of sizes it makes them at.

A case is a dict of plain values.  Lattice extents are a text "Lx x Ly x Lz x Lt" without spaces ("32x32x32x32"),
several lattices separated by commas.  Kinds:

  dslash   one application of D_oe or D_eo (the stencil alone)
  normal   one application of m^2 - D_eo D_oe
  mrhs     one D_oe on several right-hand sides
  force    the molecular-dynamics force of given X and Y, fat and (Naik) long links
  solve    canonical links and source in, canonical solution out: packing, CG, unpacking (the whole single solve)
  action   StaggeredAction forward and backward: FP64 CG, the force's gradient, unpacking
  solves   one CG call for several right-hand sides
  batch    one CG call for several lattices
"""

import torch

import paper_1612_02750_gb300 as q

C3 = -1.0 / 24.0  # Naik coefficient


def listed():
    return [
        # The smallest operator call in earnest (an 8^4 test or thermalisation lattice, FP64): launch and call latency.
        {"name": "normal_f64_8", "kind": "normal", "dims": "8x8x8x8", "prec": "f64", "naik": False, "links": "haar",
         "antiperiodic": True, "mass": 0.05},
        # A ragged, periodic lattice with links that are not unitary (smeared fat links), 16-bit, even output.
        {"name": "dslash_s16_naik_ragged", "kind": "dslash", "dims": "10x14x18x22", "prec": "f32s16", "naik": True,
         "links": "haar", "antiperiodic": False, "parity": 0},
        # The FP64 stencil at the benchmark's size: the FP64 solver and every reliable update are made of it.
        {"name": "dslash_f64_32", "kind": "dslash", "dims": "32x32x32x32", "prec": "f64", "naik": False,
         "links": "smooth", "antiperiodic": True, "parity": 1},
        # The 16-bit two-row operator at the benchmark's size: the inner iteration of the mixed solver.
        {"name": "normal_r12h_32", "kind": "normal", "dims": "32x32x32x32", "prec": "f32r12h", "naik": False,
         "links": "smooth", "antiperiodic": True, "mass": 0.01},
        # The largest operator: 64^4 with the Naik term, two-row FP32 fat and FP32 long links.
        {"name": "normal_r12_naik_64", "kind": "normal", "dims": "64x64x64x64", "prec": "f32r12", "naik": True,
         "links": "haar", "antiperiodic": True, "mass": 0.005},
        # Propagator sources: 16 right-hand sides on 24^4.
        {"name": "mrhs_r12_24_n16", "kind": "mrhs", "dims": "24x24x24x24", "prec": "f32r12", "naik": False,
         "links": "haar", "antiperiodic": True, "nrhs": 16},
        # The molecular-dynamics force with fat and long links.
        {"name": "force_naik_24", "kind": "force", "dims": "24x24x24x24", "naik": True, "links": "smooth",
         "antiperiodic": True, "force": 0},
        # The headline solve, mixed precision with 16-bit inner links, from canonical arrays and back.
        {"name": "solve_r12h_32", "kind": "solve", "dims": "32x32x32x32", "prec": "f32r12h", "naik": False,
         "links": "smooth", "antiperiodic": True, "mass": 0.01, "tol": 1e-11},
        # A small mixed solve with the Naik term (the whole lattice in the L2, latency counts).
        {"name": "solve_r12_naik_12", "kind": "solve", "dims": "12x12x12x12", "prec": "f32r12", "naik": True,
         "links": "haar", "antiperiodic": True, "mass": 0.05, "tol": 1e-11},
        # The differentiable action at the force workload's size: FP64 CG forward, force gradient backward.
        {"name": "action_f64_16", "kind": "action", "dims": "16x16x16x16", "links": "smooth", "antiperiodic": True,
         "mass": 0.05, "tol": 1e-12},
        # Propagators: 16 sources solved together.
        {"name": "solves_r12h_24_n16", "kind": "solves", "dims": "24x24x24x24", "prec": "f32r12h", "naik": False,
         "links": "haar", "antiperiodic": True, "mass": 0.05, "nrhs": 16, "tol": 1e-11},
        # Eight independent lattices, small to large, each with its own mass, solved together.
        {"name": "batch_r12h_8", "kind": "batch",
         "dims": "8x8x8x8,12x12x12x12,16x16x16x16,16x16x16x32,20x20x20x20,24x24x24x24,24x24x24x48,32x32x32x32",
         "prec": "f32r12h", "naik": False, "links": "haar", "antiperiodic": True, "mass": 0.02, "mass_to": 0.1,
         "tol": 1e-11},
    ]


def _draw_dims(rng, lo, hi, least):
    """Even extents of a lattice whose side (fourth root of the volume) is spread over lo..hi on a logarithm."""
    side = lo * (hi / lo) ** rng.random()
    while True:
        d = [max(least, 2 * round(side * 2.0 ** rng.uniform(-0.5, 0.5) / 2)) for _ in range(4)]
        v = (d[0] * d[1] * d[2] * d[3]) ** 0.25
        if lo * 0.9 <= v <= hi:
            return "x".join(str(n) for n in d)


def draw(rng):
    kind = rng.choice(["dslash", "dslash", "normal", "normal", "mrhs", "force", "solve", "solve", "action", "solves",
                       "batch"])
    naik = rng.random() < 0.5
    prec = rng.choice(["f64", "f32", "f32r12", "f32r12h", "f32s16"])
    c = {"kind": kind, "naik": naik, "prec": prec, "links": rng.choice(["haar", "smooth"]),
         "antiperiodic": rng.random() < 0.75}
    least = 4 if naik else 2
    if kind == "dslash":
        c |= {"dims": _draw_dims(rng, 4, 56, least), "parity": rng.randrange(2)}
    elif kind == "normal":
        c |= {"dims": _draw_dims(rng, 4, 48, least), "mass": round(0.005 * 20 ** rng.random(), 4)}
    elif kind == "mrhs":
        c |= {"dims": _draw_dims(rng, 6, 28, least), "nrhs": round(2 * 16 ** rng.random())}
    elif kind == "force":
        del c["prec"]
        c |= {"dims": _draw_dims(rng, 6, 36, least), "force": rng.randrange(2)}
    else:
        mass = round(0.04 * 3 ** rng.random(), 4)
        if kind == "solve":
            c |= {"dims": _draw_dims(rng, 6, 24, max(least, 4)), "mass": mass, "tol": 1e-11}
        elif kind == "action":
            del c["prec"], c["naik"]
            c |= {"dims": _draw_dims(rng, 6, 16, 4), "mass": mass, "tol": 1e-12}
        elif kind == "solves":
            c |= {"dims": _draw_dims(rng, 6, 16, max(least, 4)), "mass": mass, "nrhs": rng.randrange(2, 13),
                  "tol": 1e-11}
        else:
            n = rng.randrange(2, 7)
            c |= {"dims": ",".join(_draw_dims(rng, 6, 18, max(least, 4)) for _ in range(n)), "mass": mass,
                  "mass_to": 0.12, "tol": 1e-11}
    return c


# ------------------------------------------------------------------ inputs

def _dims(text):
    return tuple(int(n) for n in text.split("x"))


def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + stream)
    return g


def _gauss(g, shape):
    """Complex Gaussian, re and im of variance 1 (drawn in FP32, held in FP64)."""
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=g, device="cuda",
                                             dtype=torch.float32).double())


def _field(g, dims):
    lx, ly, lz, lt = dims
    return _gauss(g, (lt, lz, ly, lx, 3))


def _cross_conj(a, b):
    return torch.linalg.cross(a, b, dim=-1).conj().resolve_conj()


def _su3(g, dims, kind):
    """Canonical SU(3) links: "haar" random, or "smooth": I + 0.3 i H made unitary, H Hermitian Gaussian."""
    lx, ly, lz, lt = dims
    z = _gauss(g, (lt, lz, ly, lx, 4, 3, 3))
    if kind == "smooth":
        z = 0.075j * (z + z.mH)  # 0.3 i H, H = sum of Gell-Mann matrices / 2 with unit Gaussian weights (plus a trace)
        z += torch.eye(3, dtype=z.dtype, device=z.device)
    a, b = z[..., 0, :], z[..., 1, :]
    a = a / a.abs().square().sum(-1, keepdim=True).sqrt()
    for _ in range(2):
        b = b - (a.conj() * b).sum(-1, keepdim=True) * a
        b = b / b.abs().square().sum(-1, keepdim=True).sqrt()
    z[..., 0, :], z[..., 1, :], z[..., 2, :] = a, b, _cross_conj(a, b)
    return z


def _long(g, dims):
    """Long links: complex Gaussian over sqrt 3 (not unitary)."""
    lx, ly, lz, lt = dims
    return _gauss(g, (lt, lz, ly, lx, 4, 3, 3)) * 3.0 ** -0.5


def _links(case, dims, seed, k=0):
    """Canonical fat and long (or None) links of the k-th lattice of a case."""
    u = _su3(_gen(seed, 10 * k), dims, case["links"])
    return u, (_long(_gen(seed, 10 * k + 1), dims) if case.get("naik") else None)


def _masses(case, n):
    lo, hi = case["mass"], case["mass_to"]
    return [lo * (hi / lo) ** (k / max(1, n - 1)) for k in range(n)]


def _inner(lat, prec, u64, w64):
    """The inner copies of a mixed solve."""
    if prec == "f64":
        return None, None
    return (q.qex_convert_links(lat, "f64", u64, prec),
            None if w64 is None else q.qex_convert_links(lat, "f64", w64, q.qex_long_links_prec(prec)))


def prepare(case, seed):
    kind, dims = case["kind"], [_dims(t) for t in case["dims"].split(",")]
    if kind == "batch":
        items = []
        for k, (d, m) in enumerate(zip(dims, _masses(case, len(dims)))):
            lat = q.Lattice(d, case["antiperiodic"])
            u, w = _links(case, d, seed, k)
            u64 = q.qex_pack_links(lat, "f64", u)
            w64 = None if w is None else q.qex_pack_links(lat, "f64", w)
            u32, w32 = _inner(lat, case["prec"], u64, w64)
            items.append({"lat": lat, "fat64": u64, "lng64": w64, "fat32": u32, "lng32": w32, "c_naik": C3, "mass": m,
                          "b64": q.qex_pack_field(lat, "f64", 0, _field(_gen(seed, 10 * k + 2), d))})
        return {"case": case, "items": items}
    dims = dims[0]
    lat = q.Lattice(dims, case["antiperiodic"])
    s = {"case": case, "lat": lat}
    u, w = _links(case, dims, seed)
    if kind == "solve":
        return s | {"u": u, "w": w, "b": _field(_gen(seed, 2), dims)}
    if kind == "action":
        return s | {"u": u.requires_grad_(True), "b": _field(_gen(seed, 2), dims)}
    if kind == "force":
        return s | {"fat": q.qex_pack_links(lat, "f64", u), "lng": None if w is None else q.qex_pack_links(lat, "f64", w),
                    "x": q.qex_pack_field(lat, "f64", 0, _field(_gen(seed, 2), dims)),
                    "y": q.qex_pack_field(lat, "f64", 1, _field(_gen(seed, 3), dims))}
    if kind == "solves":
        u64 = q.qex_pack_links(lat, "f64", u)
        w64 = None if w is None else q.qex_pack_links(lat, "f64", w)
        u32, w32 = _inner(lat, case["prec"], u64, w64)
        b = torch.cat([q.qex_pack_field(lat, "f64", 0, _field(_gen(seed, 2 + 10 * r), dims))
                       for r in range(case["nrhs"])])
        return s | {"fat64": u64, "lng64": w64, "fat32": u32, "lng32": w32, "b64": b}
    prec = case["prec"]
    s["fat"] = q.qex_pack_links(lat, prec, u)
    s["lng"] = None if w is None else q.qex_pack_links(lat, q.qex_long_links_prec(prec), w)
    del u, w
    if kind == "mrhs":
        s["in"] = torch.cat([q.qex_pack_field(lat, prec, 0, _field(_gen(seed, 2 + 10 * r), dims))
                             for r in range(case["nrhs"])])
        s["out"] = q.empty_fields(lat, prec, case["nrhs"])
        return s
    s["in"] = q.qex_pack_field(lat, prec, 1 - case.get("parity", 0) if kind == "dslash" else 0,
                               _field(_gen(seed, 2), dims))
    s["out"], s["tmp"] = q.empty_field(lat, prec), q.empty_field(lat, prec)
    return s


# ---------------------------------------------------------------- one pass

def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "dslash":
        return q.qex_dslash(s["lat"], c["prec"], s["fat"], s["lng"], C3, c["parity"], s["in"], s["out"])
    if kind == "normal":
        return q.qex_normal_op(s["lat"], c["prec"], s["fat"], s["lng"], C3, c["mass"], s["in"], s["out"], s["tmp"])
    if kind == "mrhs":
        return q.qex_dslash_mrhs(s["lat"], c["prec"], s["fat"], s["lng"], C3, 1, c["nrhs"], s["in"], s["out"])
    if kind == "force":
        return q.qex_force(s["lat"], s["fat"], s["lng"], C3, s["x"], s["y"], kind=c["force"])
    if kind == "solve":
        lat, prec = s["lat"], c["prec"]
        u32 = w64 = w32 = None
        if prec == "f64":
            u64 = q.qex_pack_links(lat, "f64", s["u"])
            if s["w"] is not None:
                w64 = q.qex_pack_links(lat, "f64", s["w"])
        else:
            u64, u32 = q.qex_pack_links_pair(lat, s["u"], prec)
            if s["w"] is not None:
                w64, w32 = q.qex_pack_links_pair(lat, s["w"], q.qex_long_links_prec(prec))
        b = q.qex_pack_field(lat, "f64", 0, s["b"])
        x = torch.zeros_like(b)
        q.qex_cg(lat, prec, u64, w64, u32, w32, C3, c["mass"], b, x, tol=c["tol"], delta=0.01)
        return q.qex_unpack_field(lat, "f64", 0, x)
    if kind == "action":
        s["u"].grad = None
        a = q.StaggeredAction.apply(s["u"], None, s["b"], s["lat"], c["mass"], 0.0, "f64", c["tol"])
        a.backward()
        return a.detach(), s["u"].grad
    if kind == "solves":
        x = torch.zeros_like(s["b64"])
        q.qex_cg_mrhs(s["lat"], c["prec"], s["fat64"], s["lng64"], s["fat32"], s["lng32"], C3, c["mass"], c["nrhs"],
                      s["b64"], x, tol=c["tol"], delta=0.01)
        return x
    xs = [torch.zeros_like(it["b64"]) for it in s["items"]]
    q.qex_cg_batch([it | {"x64": x} for it, x in zip(s["items"], xs)], c["prec"], tol=c["tol"], delta=0.01)
    return xs


# -------------------------------------------------------------- what it costs

_LINK = {"f64": 144, "f32": 72, "f32r12": 48, "f32r12h": 24, "f32s16": 40}  # bytes of one link
_LONG = {"f64": "f64", "f32": "f32", "f32r12": "f32", "f32r12h": "f32s16", "f32s16": "f32s16"}


def _apply(case, prec, vh, nrhs=1):
    """One Dslash: its 8 (16) links a site once, each vector in once, each vector out once; the usual flop count."""
    vec = 48 if prec == "f64" else 24
    links = 8 * _LINK[prec] + (8 * _LINK[_LONG[prec]] if case.get("naik") else 0)
    return vh * (links + 2 * nrhs * vec), vh * nrhs * (1146 if case.get("naik") else 570)


def _iterations(case, dims, mass):
    """CG iterations to the tolerance, roughly: in proportion to 1/m on Haar links, bounded by the free spectrum's
    gap (the smallest antiperiodic momentum) on smooth ones."""
    n = 65.0 / mass * (1.2 if case["tol"] < 5e-12 else 1.0)
    if case["links"] == "smooth":
        n = min(n, 8.0 * max(dims))
    return n


def _cg(case, dims, mass, nrhs=1):
    """Two operator applications an iteration in the inner precision, and the vector updates (x, r, p: three read and
    written, A p read)."""
    vh = dims[0] * dims[1] * dims[2] * dims[3] // 2
    prec = case.get("prec", "f64")
    b, f = _apply(case, prec, vh, nrhs)
    n = _iterations(case, dims, mass)
    return n * (2 * b + 7 * nrhs * vh * (48 if prec == "f64" else 24)), n * (2 * f + 36 * nrhs * vh)


def work(case):
    kind, lats = case["kind"], [_dims(t) for t in case["dims"].split(",")]
    d = lats[0]
    vh = d[0] * d[1] * d[2] * d[3] // 2
    if kind in ("dslash", "normal", "mrhs"):
        b, f = _apply(case, case["prec"], vh, case.get("nrhs", 1))
        if kind == "normal":
            b, f = 2 * b, 2 * f + 12 * vh
    elif kind == "force":  # X and Y in; F out, and the links in where F needs them; both sets with the Naik term
        sets = 2 if case["naik"] else 1
        b = 2 * 48 * vh + sets * 8 * vh * 144 * (2 if case["force"] == 0 else 1)
        f = sets * 8 * vh * (66 + 36 + 36 if case["force"] == 0 else 42)
    elif kind == "solve":
        b, f = _cg(case, d, case["mass"])
        sets = 2 if case["naik"] else 1
        b += sets * 8 * vh * 2 * 144 + 2 * vh * 4 * 48  # canonical links to internal ones, b and x
    elif kind == "action":
        b, f = _cg(case, d, case["mass"])
        b += 4 * 8 * vh * 144 + 4 * vh * 48
    elif kind == "solves":
        b, f = _cg(case, d, case["mass"], case["nrhs"])
    else:
        parts = [_cg(case, e, m) for e, m in zip(lats, _masses(case, len(lats)))]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------- the same in 64 bits

class _Plain:
    """The operator from its definition, in complex128 torch on even-odd half fields [Vh, 3]."""

    def __init__(self, dims, antiperiodic):
        self.dims, self.anti = dims, antiperiodic
        lx, ly, lz, lt = dims
        lex = torch.arange(lx * ly * lz * lt, device="cuda")
        x, y, z, t = lex % lx, lex // lx % ly, lex // (lx * ly) % lz, lex // (lx * ly * lz)
        par = (x + y + z + t) % 2
        self.site, self.c = [], []
        for p in (0, 1):
            self.site.append(lex[par == p])
            self.c.append([v[par == p] for v in (x, y, z, t)])

    def hop(self, p, mu, k):
        """Even-odd index of site + k mu for the sites of parity p."""
        c = list(self.c[p])
        c[mu] = (c[mu] + k) % self.dims[mu]
        lx, ly, lz, _ = self.dims
        return (c[0] + lx * (c[1] + ly * (c[2] + lz * c[3]))) // 2

    def sign(self, p, mu, k):
        """Phase and boundary sign of the k-step link leaving the sites of parity p along +mu."""
        c = self.c[p]
        s = 1.0 - 2.0 * (sum(c[:mu]) % 2).double() if mu else torch.ones(len(c[0]), dtype=torch.float64, device="cuda")
        if mu == 3 and self.anti:
            s = torch.where(c[3] + k >= self.dims[3], -s, s)
        return s

    def half(self, lex_array, p):
        """The parity-p part of a canonical array."""
        return lex_array.reshape((-1,) + tuple(lex_array.shape[4:]))[self.site[p]]

    def terms(self, u, w, p):
        """(matrix [Vh, 3, 3], index [Vh]) of each hop of D_{p,1-p}; u and w: canonical links, or None."""
        for links, coef, k in ((u, 1.0, 1), (w, C3, 3)):
            if links is None:
                continue
            for mu in range(4):
                here, there = self.half(links[..., mu, :, :], p), self.half(links[..., mu, :, :], 1 - p)
                j = self.hop(p, mu, k)
                yield coef * self.sign(p, mu, k)[:, None, None] * here, j
                j = self.hop(p, mu, -k)
                yield -coef * (self.sign(1 - p, mu, k)[:, None, None] * there)[j].mH, j

    def dslash(self, u, w, p, psi):
        """D_{p,1-p} psi for psi [Vh, 3, n]."""
        out = torch.zeros_like(psi)
        for m, j in self.terms(u, w, p):
            out += m @ psi[j]
        return out

    def solve(self, u, w, mass, b):
        """(m^2 - D_eo D_oe)^-1 b for b [Vh, 3, n], by CG on all n at once."""
        ops = []
        for p in (0, 1):
            t = list(self.terms(u, w, p))
            ops.append((torch.cat([m for m, _ in t], -1), torch.stack([j for _, j in t], 1)))
            del t

        def d(p, v):
            m, j = ops[p]
            g = v[j].reshape(len(v), -1, v.shape[-1])
            if v.shape[-1] == 1:
                return (m * g.transpose(1, 2)).sum(-1, keepdim=True)
            return m @ g

        def dot(a, c):
            return (a.conj() * c).real.sum((0, 1))

        x, r = torch.zeros_like(b), b.clone()
        v, rr = r.clone(), dot(r, r)
        stop = 1e-28 * rr
        for k in range(20000):
            av = mass * mass * v - d(0, d(1, v))
            a = rr / dot(v, av)
            x += a * v
            r -= a * av
            new = dot(r, r)
            v = r + (new / rr) * v
            rr = new
            if k % 16 == 0 and bool((rr <= stop).all()):
                break
        return x


def _stored(links, prec):
    """The values that a link set of format prec holds (row 2 of the two-row formats rebuilt in 64 bits)."""
    if prec == "f64" or links is None:
        return links
    if prec == "f32":
        return links.to(torch.complex64).to(torch.complex128)
    if prec == "f32s16":
        v = torch.view_as_real(links)
        big = v.abs().amax((-3, -2, -1), keepdim=True) / 32767.0
        step = big.float()
        step = torch.where(step.double() < big, torch.nextafter(step, torch.full_like(step, float("inf"))), step)
        step = step.double()
        return torch.view_as_complex((v * (1.0 / step)).round().clamp(-32767, 32767) * step)
    if prec == "f32r12":
        z = links.to(torch.complex64).to(torch.complex128)
    else:
        z = torch.view_as_complex((torch.view_as_real(links) * 32767.0).round().clamp(-32767, 32767) / 32767.0)
    z[..., 2, :] = _cross_conj(z[..., 0, :], z[..., 1, :])
    return z


def _round(v, prec):
    return v if prec == "f64" else v.to(torch.complex64).to(torch.complex128)


def _planes(v, prec):
    """A half field [Vh, 3] as the internal layout holds it, in 64 bits."""
    if prec == "f64":
        return torch.view_as_real(v.T.contiguous()).reshape(-1)
    return torch.cat([torch.view_as_real(v[:, :2].contiguous()).reshape(-1),
                      torch.view_as_real(v[:, 2].contiguous()).reshape(-1)])


def _outer(plain, p, mu, k, x, y):
    """G_mu on the sites of parity p: s Y(x+k mu) X(x)^+ on even, -s X(x+k mu) Y(x)^+ on odd sites."""
    here, there = (x, y) if p == 0 else (y, x)
    s = plain.sign(p, mu, k) * (1.0 if p == 0 else -1.0)
    return s[:, None, None] * there[plain.hop(p, mu, k)][:, :, None] * here[:, None, :].conj()


def _force(plain, links, coef, k, x, y, kind):
    blocks = []
    for p in (0, 1):
        for mu in range(4):
            m = coef * _outer(plain, p, mu, k, x, y)
            if kind == 1:
                m = 2.0 * m.mH
            else:
                m = plain.half(links[..., mu, :, :], p) @ m
                m = m - m.mH
                m = m - torch.diagonal(m, dim1=-2, dim2=-1).mean(-1)[:, None, None] * torch.eye(3, device="cuda")
            blocks.append(torch.view_as_real(m.reshape(-1, 9).T.contiguous()).reshape(-1))
    return torch.cat(blocks)


def exact(case, seed):
    kind, lats = case["kind"], [_dims(t) for t in case["dims"].split(",")]
    if kind == "batch":
        out = []
        for k, (d, m) in enumerate(zip(lats, _masses(case, len(lats)))):
            plain = _Plain(d, case["antiperiodic"])
            u, w = _links(case, d, seed, k)
            b = plain.half(_field(_gen(seed, 10 * k + 2), d), 0)
            out.append(_planes(plain.solve(u, w, m, b[..., None])[..., 0], "f64"))
        return out
    d = lats[0]
    plain = _Plain(d, case["antiperiodic"])
    u, w = _links(case, d, seed)
    if kind in ("dslash", "normal", "mrhs"):
        prec = case["prec"]
        u, w = _stored(u, prec), _stored(w, _LONG[prec])
        if kind == "dslash":
            p = case["parity"]
            v = _round(plain.half(_field(_gen(seed, 2), d), 1 - p), prec)
            return _planes(plain.dslash(u, w, p, v[..., None])[..., 0], prec)
        if kind == "normal":
            v = _round(plain.half(_field(_gen(seed, 2), d), 0), prec)[..., None]
            return _planes((case["mass"] ** 2 * v - plain.dslash(u, w, 0, plain.dslash(u, w, 1, v)))[..., 0], prec)
        v = torch.stack([_round(plain.half(_field(_gen(seed, 2 + 10 * r), d), 0), prec) for r in range(case["nrhs"])],
                        -1)
        v = plain.dslash(u, w, 1, v)
        return torch.cat([_planes(v[..., r], prec) for r in range(case["nrhs"])])
    if kind == "force":
        x, y = plain.half(_field(_gen(seed, 2), d), 0), plain.half(_field(_gen(seed, 3), d), 1)
        return (_force(plain, u, 1.0, 1, x, y, case["force"]),
                None if w is None else _force(plain, w, C3, 3, x, y, case["force"]))
    if kind == "solves":
        b = torch.stack([plain.half(_field(_gen(seed, 2 + 10 * r), d), 0) for r in range(case["nrhs"])], -1)
        x = plain.solve(u, w, case["mass"], b)
        return torch.cat([_planes(x[..., r], "f64") for r in range(case["nrhs"])])
    field = _field(_gen(seed, 2), d)
    b = plain.half(field, 0)[..., None]
    x = plain.solve(u, w, case["mass"], b)
    if kind == "solve":
        out = torch.zeros_like(field)
        out.view(-1, 3)[plain.site[0]] = x[..., 0]
        return out
    y = plain.dslash(u, None, 1, x)
    grad = torch.zeros_like(u)
    g = grad.view(-1, 4, 3, 3)
    for p in (0, 1):
        for mu in range(4):
            g[plain.site[p], mu] = 2.0 * _outer(plain, p, mu, 1, x[..., 0], y[..., 0]).mH
    return (b.conj() * x).real.sum(), grad
