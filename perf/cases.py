"""The work that users of this library have it do, as cases for timing and comparison.

Five kinds, all through the package's public entry points:

  product  y = A p with a context that is kept (dda_matvec, dda_matvec_batch): complex64, double-float and complex128
  solve    incident fields, Krylov solves and cross sections of a batch of incidences on one target
  gradient a solve and its adjoint: cross sections, per-dipole and per-material permittivity gradients
  setup    a target's mask and materials to a context with its tensor spectrum and ranks
  observe  incident fields and cross sections alone, on given dipole moments

Targets are ellipsoids that fill their box (spheres in cubic boxes), whole boxes with spherical inclusions, and porous
clusters of small spheres.  Lattices go from a few sites to 256^3, ragged ones among them; `exact` restates the method
with plain FFTs in 64 bits.
"""
import math

import numpy as np
import torch

import paper_0908_0863_gb300 as dda

DEV = "cuda"
M_WATER, M_GLASS, M_SOOT = (1.33, 0.05), (1.5, 0.01), (1.7, 0.1)
M_AGGREGATE, M_INCLUSION, M_HOST = (1.6, 0.05), (2.0, 0.5), (1.33, 0.001)
COST = {"c64": 1, "c128df": 12, "c128": 28}   # of one product, in complex64 products of the same lattice
METHODS = ("bicgstab", "qmr", "bicg_sym", "qmr_sym", "tfqmr", "rbicgstab2", "mlbicgstab2")


def _case(kind, shape, target="ellipsoid", m=(M_WATER,), mkd=0.5, rule="cmrr", nb=1, **more):
    """A case as plain values: lattice K x J x P, refractive indices (one or two), |m| k d of the denser material."""
    m1 = m[1] if len(m) > 1 else m[0]
    return {"kind": kind, "K": shape[0], "J": shape[1], "P": shape[2], "target": target, "nmat": len(m),
            "m0_re": m[0][0], "m0_im": m[0][1], "m1_re": m1[0], "m1_im": m1[1], "mkd": mkd, "rule": rule, "nb": nb, **more}


def listed():
    ell2 = {"m": (M_GLASS, M_SOOT), "mkd": 0.8, "rule": "ldr"}
    cases = [
        # the smallest target of a parameter scan: launches and latency are all of it
        ("product_c64_16", _case("product", (16, 16, 16), dtype="c64")),
        # an ordinary product: two-material LDR ellipsoid, as in a mixed solve's inner iterations
        ("product_c64_128", _case("product", (128, 128, 128), dtype="c64", **ell2)),
        # the largest: a water sphere on the 256^3 lattice, padded to 512^3
        ("product_c64_256", _case("product", (256, 256, 256), dtype="c64")),
        # many orientations of one sparse aggregate on a ragged lattice (3 * 2^a and 5 * 2^a lines)
        ("product_c64_cluster_b32", _case("product", (92, 72, 80), "spheres", (M_AGGREGATE,), nb=32, dtype="c64")),
        # the mixed refinement's true residuals: double-float products of complex128 vectors
        ("product_df_128", _case("product", (128, 128, 128), dtype="c128df", **ell2)),
        # an FP64 product on a ragged lattice, as in the FP64 solves
        ("product_c128_75x60x50", _case("product", (75, 60, 50), dtype="c128", **ell2)),
        # one large mixed-precision solve, the library's main use
        ("solve_mixed_128", _case("solve", (128, 128, 128), method="bicgstab", precision="mixed", tol=1e-8, products=315)),
        # orientation averaging: many incidences on one aggregate in lock step
        ("solve_mixed_cluster_b32", _case("solve", (62, 54, 46), "spheres", (M_AGGREGATE,), nb=32, method="bicgstab",
                                          precision="mixed", tol=1e-8, products=60)),
        # a small FP64 solve in the paper's form: point-Jacobi, complex-symmetric BiCG, 1e-10
        ("solve_fp64_jacobi_32", _case("solve", (32, 32, 32), m=(M_GLASS, M_SOOT), rule="ldr", method="bicg_sym+jacobi",
                                       precision="fp64", tol=1e-10, products=96)),
        # forward and adjoint solve of the inclusion cube: material gradients of C_abs
        ("gradient_inclusions_48", _case("gradient", (48, 48, 48), "box", (M_HOST, M_INCLUSION), method="bicgstab",
                                         precision="mixed", tol=1e-8, products=300)),
        # a new target or wavelength: bit fields, ranks and the tensor spectrum of the 100^3 cube
        ("setup_box_100", _case("setup", (100, 100, 100), "box", (M_HOST, M_INCLUSION))),
        # incident fields and cross sections of two polarisations on the paper's 200^3 sphere
        ("observe_sphere_200", _case("observe", (200, 200, 200), nb=2)),
    ]
    return [dict(c, name=n) for n, c in cases]


def _edges(rng, lo, hi, most):
    """Three edges, log-uniform in [lo, hi], odd ones among them, of at most `most` padded points."""
    while True:
        e = [int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) for _ in range(3)]
        if math.prod(_padded(n) for n in e) <= most:
            return e


def draw(rng):
    """One more case: kinds, sizes, materials, types and methods over the whole ranges."""
    kind = rng.choice(("product", "product", "product", "solve", "gradient", "setup", "observe"))
    target = rng.choice(("ellipsoid", "ellipsoid", "box", "spheres"))
    two = rng.random() < 0.5
    m = (M_HOST, M_INCLUSION) if target == "box" else (M_GLASS, M_SOOT) if two else rng.choice(((M_WATER,), (M_AGGREGATE,)))
    base = {"target": target, "m": m, "mkd": rng.choice((0.3, 0.5)), "rule": rng.choice(("cmrr", "ldr"))}
    if kind == "product":
        dtype = rng.choice(("c64", "c64", "c64", "c128df", "c128"))
        nb = rng.choice((1, 1, 2, 5, 16, 32))
        return _case(kind, _edges(rng, 4, 256, 2**27 // (COST[dtype] * nb)), nb=nb, dtype=dtype, **base)
    if kind == "solve":
        precision = rng.choice(("mixed", "mixed", "fp64"))
        nb, jacobi = rng.choice((1, 2, 8, 32)), rng.choice(("", "+jacobi"))
        most = 2**23 // nb if precision == "mixed" else 2**18 // nb
        return _case(kind, _edges(rng, 4, 128, max(most, 2**12)), nb=nb, method=rng.choice(METHODS) + jacobi, precision=precision,
                     tol=1e-8, products=20, **base)
    if kind == "gradient":
        return _case(kind, _edges(rng, 4, 64, 2**20), method="bicgstab", precision=rng.choice(("mixed", "fp64")), tol=1e-8,
                     products=40, **base)
    if kind == "setup":
        return _case(kind, _edges(rng, 4, 160, 2**24), **base)
    return _case(kind, _edges(rng, 8, 256, 2**26), nb=rng.choice((1, 2, 8)), **base)


# ---------------------------------------------------------------- targets

def _shape(case):
    return case["K"], case["J"], case["P"]


def _padded(n):
    """Length of the circulant extension of n points: the smallest 2^a, 3 * 2^a or 5 * 2^a (a >= 3) of at least 2n - 1."""
    best = 0
    for length in (2, 24, 40):
        while length < 2 * n - 1:
            length *= 2
        best = length if not best else min(best, length)
    return best


def _rng(case, salt, seed=0):
    return np.random.Generator(np.random.PCG64([case["K"], case["J"], case["P"], salt, seed]))


def _axes(case, device):
    """Site indices along z, y, x, broadcastable over a [P][J][K] volume."""
    K, J, P = _shape(case)
    a = [torch.arange(n, dtype=torch.float64, device=device) for n in (P, J, K)]
    return a[0][:, None, None], a[1][None, :, None], a[2][None, None, :]


def _ball(case, device, g, volume, rmin, rmax, fraction):
    """Adds balls of radius [rmin, rmax] at uniform centres to a boolean volume until the fraction of it is covered."""
    z, y, x = _axes(case, device)
    K, J, P = _shape(case)
    for count in range(1, 4097):
        r, cx, cy, cz = g.uniform(rmin, rmax), g.uniform(0, K), g.uniform(0, J), g.uniform(0, P)
        lo = [max(0, int(c - r) - 1) for c in (cz, cy, cx)]
        s = tuple(slice(a, a + 2 * int(r) + 4) for a in lo)
        near = ((z[s[0]] + 0.5 - cz) ** 2 + (y[:, s[1]] + 0.5 - cy) ** 2 + (x[:, :, s[2]] + 0.5 - cx) ** 2) <= r * r
        volume[s] |= near
        if count % 16 == 0 and float(volume.sum()) >= fraction * volume.numel():
            break
    return volume


def _mask(case, device):
    """The occupied sites of the case's target, bool [P][J][K] (the same for every seed)."""
    K, J, P = _shape(case)
    if case["target"] == "box":
        return torch.ones((P, J, K), dtype=torch.bool, device=device)
    if case["target"] == "spheres":
        v = torch.zeros((P, J, K), dtype=torch.bool, device=device)
        v[P // 2, J // 2, K // 2] = True
        return _ball(case, device, _rng(case, 1), v, 4.0, 4.0, 0.06)
    z, y, x = _axes(case, device)
    return ((2 * z + 1 - P) / P) ** 2 + ((2 * y + 1 - J) / J) ** 2 + ((2 * x + 1 - K) / K) ** 2 <= 1.0


def _materials(case, device):
    """Material index per site, uint8 [P][J][K]: inclusions in a box, else 30 % of the second at random."""
    K, J, P = _shape(case)
    if case["nmat"] == 1:
        return torch.zeros((P, J, K), dtype=torch.uint8, device=device)
    if case["target"] == "box":
        v = torch.zeros((P, J, K), dtype=torch.bool, device=device)
        return _ball(case, device, _rng(case, 2), v, 3.0, 6.0, 0.2).to(torch.uint8)
    u = _rng(case, 3).random(P * J * K, dtype=np.float32).reshape(P, J, K)
    return (torch.from_numpy(u).to(device) < 0.3).to(torch.uint8)


def _refr(case):
    m = [complex(case["m0_re"], case["m0_im"]), complex(case["m1_re"], case["m1_im"])]
    return m[: case["nmat"]]


def _k(case):
    return case["mkd"] / max(abs(m) for m in _refr(case))


KHAT, E0 = (0.0, 0.0, 1.0), (1.0, 0.0, 0.0)   # of the LDR polarisabilities


def _directions(case, seed):
    """nb incidences: direction uniform on the sphere, a real polarisation across it."""
    g, out = _rng(case, 4, seed), []
    for _ in range(case["nb"]):
        kh = g.normal(size=3)
        kh /= np.linalg.norm(kh)
        e = np.cross(kh, g.normal(size=3))
        out.append((kh, e / np.linalg.norm(e)))
    return out


def _normal(case, salt, seed, shape):
    """Circular complex normal vectors, complex128 on the device."""
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * seed + salt)
    return torch.randn(shape, dtype=torch.complex128, device=DEV, generator=g)


def _bits(case):
    """The packed target: occupancy words and, for two materials, composition words, on the device."""
    mask = _mask(case, DEV).to(torch.uint8).reshape(-1)
    bits = torch.empty((mask.numel() + 31) // 32, dtype=torch.int32, device=DEV)
    dda.dda_pack_occupancy(mask, bits)
    comp = None
    if case["nmat"] > 1:
        mats = _materials(case, DEV).reshape(-1, 1).expand(-1, 3).contiguous()
        comp = torch.empty((3 * mask.numel() + 31) // 32, dtype=torch.int32, device=DEV)
        dda.dda_pack_composition(mats, mask.numel(), case["nmat"], comp)
    return bits, comp


def _lattice(case):
    bits, comp = _bits(case)
    alpha = dda.dda_polarizability(_refr(case), _k(case), case["rule"], KHAT, E0)
    return dda.Lattice(_shape(case), bits, alpha, _k(case), comp, case["nmat"])


# ---------------------------------------------------------------- cases

def prepare(case, seed):
    kind, nb = case["kind"], case["nb"]
    if kind == "setup":
        K, J, P = _shape(case)
        half = [_padded(n) // 2 + 1 for n in (J, K, P)]
        mats = _materials(case, DEV).reshape(-1, 1).expand(-1, 3).contiguous()
        return {"case": case, "mask": _mask(case, DEV).to(torch.uint8).reshape(-1), "mats": mats,
                # another wavelength for every seed
                "k": _k(case) * (1.0 + 0.01 * (seed % 16)),
                "ranks": torch.empty(K * J * P, dtype=torch.int32, device=DEV),
                "spectrum": torch.empty((*half, 6), dtype=torch.complex128, device=DEV)}
    lat = _lattice(case)
    state = {"case": case, "lat": lat, "inc": _directions(case, seed)}
    shape = (nb, 3, lat.n_dipoles)
    if kind == "product":
        p = _normal(case, 5, seed, shape)
        state["p"] = p.to(torch.complex64) if case["dtype"] == "c64" else p
        state["y"] = torch.empty_like(state["p"])
    elif kind == "observe":
        # moments near the polarisability times the field
        E = torch.empty(shape, dtype=torch.complex128, device=DEV)
        for b, (kh, e) in enumerate(state["inc"]):
            lat.incident_field(kh, e, E[b])
        state["P"] = 0.05 * E * (1.0 + 0.2j) + 0.01 * _normal(case, 6, seed, shape)
        state["E"] = E
    else:
        state["E"] = torch.empty(shape, dtype=torch.complex128, device=DEV)
        state["P"] = torch.empty_like(state["E"])
        lat.reserve(nb, case["precision"])
        if kind == "gradient":
            state["dalpha"] = dda.dda_polarizability_derivative(_refr(case), _k(case), case["rule"], KHAT, E0)
            state["grad"] = torch.empty(lat.n_dipoles, dtype=torch.complex128, device=DEV)
    torch.cuda.synchronize()
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "setup":
        n, mask = state["mask"].numel(), state["mask"]
        bits = torch.empty((n + 31) // 32, dtype=torch.int32, device=DEV)
        dda.dda_pack_occupancy(mask, bits)
        comp = None
        if case["nmat"] > 1:
            comp = torch.empty((3 * n + 31) // 32, dtype=torch.int32, device=DEV)
            dda.dda_pack_composition(state["mats"], n, case["nmat"], comp)
        alpha = dda.dda_polarizability(_refr(case), state["k"], case["rule"], KHAT, E0)
        with dda.Lattice(_shape(case), bits, alpha, state["k"], comp, case["nmat"]) as lat:
            lat.site_ranks(state["ranks"])
            lat.tensor_spectrum(state["spectrum"])
        return {"bits": bits, "ranks": state["ranks"], "spectrum": state["spectrum"]}
    lat = state["lat"]
    if kind == "product":
        dda.dda_matvec_batch(lat.ctx, state["p"], state["y"], dtype="c128df" if case["dtype"] == "c128df" else None)
        return state["y"]
    E, P = state["E"], state["P"]
    for b, (kh, e) in enumerate(state["inc"]):
        lat.incident_field(kh, e, E[b])
    if kind == "observe":
        return {"E": E, "cross": lat.cross_sections_batch(E, P)}
    args = (case["method"], case["precision"], case["tol"], 4000)
    status, _, info = lat.solve_batch(E, P, *args)
    if status != dda.DDA_OK:
        raise RuntimeError(f"solve: {status} {info}")
    cross = lat.cross_sections_batch(E, P)
    if kind == "solve":
        return {"P": P, "cross": cross}
    status, info = lat.gradient("abs", E[0], P[0], state["dalpha"], state["grad"], *args)
    if status != dda.DDA_OK:
        raise RuntimeError(f"adjoint solve: {status} {info}")
    return {"P": P, "cross": cross, "grad": state["grad"], "sums": dda.dda_material_sums(lat.ctx, state["grad"], case["nmat"])}


# ---------------------------------------------------------------- work

def _product_work(case, elem):
    """One product: the flops of the pruned line transforms (5 L log2 L each) and of the 3 x 3 spectrum product, and
    the bytes of the vectors, the half spectrum and the bit field."""
    (K, J, P), nd = _shape(case), int(_mask(case, DEV if torch.cuda.is_available() else "cpu").sum())
    Lx, Ly, Lz = (_padded(n) for n in (K, J, P))

    def line(length):
        return 5 * length * math.log2(length)

    flops = 6 * (K * P * line(Ly) + Ly * P * line(Lx) + Lx * Ly * line(Lz)) + 84 * Lx * Ly * Lz
    spectrum = 6 * (Lx // 2 + 1) * (Ly // 2 + 1) * (Lz // 2 + 1) * elem
    return nd, flops, spectrum, K * J * P / 8


def work(case):
    kind, nb = case["kind"], case["nb"]
    elem = 8 if case.get("dtype") == "c64" or case.get("precision") == "mixed" else 16
    nd, flops, spectrum, bits = _product_work(case, elem)
    sites = case["K"] * case["J"] * case["P"]
    if kind == "product":
        return {"bytes": 6 * nd * elem * nb + spectrum + bits, "flops": flops * nb}
    if kind == "setup":
        out = spectrum / elem * 16
        Lx, Ly, Lz = (_padded(n) for n in _shape(case))
        lines = (case["J"] * case["P"] * 5 * Lx * math.log2(Lx) + (Lx // 2 + 1) * case["P"] * 5 * Ly * math.log2(Ly)
                 + (Lx // 2 + 1) * (Ly // 2 + 1) * 5 * Lz * math.log2(Lz))
        return {"bytes": out + 9 * sites, "flops": 6 * lines + 100 * sites}
    if kind == "observe":
        return {"bytes": nb * 3 * 3 * nd * 16 + bits, "flops": nb * nd * 60}
    # solves: `products` per right-hand side is about what the method needs on such a target; the fields go in and the
    # moments come out in complex128
    vectors = 2 * 3 * nd * 16 * nb + (nd * 16 if kind == "gradient" else 0)
    return {"bytes": vectors + spectrum + bits, "flops": case["products"] * nb * (flops + 100 * nd)}


def tolerance(case):
    kind = case["kind"]
    if kind == "product":
        # FP32, 48-bit and 53-bit transforms of up to 512-point lines: four times the error against 64 bits
        return {"rel": {"c64": 8e-7, "c128df": 1.5e-14, "c128": 2e-15}[case["dtype"]]}
    if kind == "setup":
        return {"rel": 2e-15}
    if kind == "observe":
        return {"rel": 2e-14}   # phases of up to a few hundred radians
    # two solutions of the same residual tolerance: that times the condition of the system
    return {"rel": 12 * case["tol"]}


# ---------------------------------------------------------------- 64 bits, plain torch

def _alpha_inverse(case, k, derivative=False):
    """1/alpha per material, or its derivative by the permittivity: Clausius-Mossotti with radiative reaction, or the
    lattice dispersion relation (Draine and Goodman 1993)."""
    out = []
    for m in _refr(case):
        eps = m * m
        s = sum((complex(a) * b) ** 2 for a, b in zip(KHAT, E0)).real
        if derivative:
            d = -4 * math.pi / (eps - 1) ** 2
            out.append(d + (0.1648469 - 1.7700004 * s) * k * k if case["rule"] == "ldr" else d)
            continue
        inv = 4 * math.pi / 3 * (eps + 2) / (eps - 1) - 2j / 3 * k**3
        if case["rule"] == "ldr":
            inv += (-1.8915316 + eps * (0.1648469 - 1.7700004 * s)) * k * k
        out.append(inv)
    return torch.tensor(out, dtype=torch.complex128, device=DEV)


class _Exact:
    """The interaction matrix of a case by unpruned FFTs of the whole padded lattice."""

    def __init__(self, case, k, with_target=True):
        self.n = _shape(case)[::-1]
        self.L = tuple(_padded(v) for v in self.n)
        grids, inside = [], None
        for axis, (n, L) in enumerate(zip(self.n, self.L)):
            i = torch.arange(L, dtype=torch.float64, device=DEV)
            d = torch.where(i < n, i, i - L)
            view = [1, 1, 1]
            view[axis] = L
            ok = ((i < n) | (i > L - n)).view(view)
            inside = ok if inside is None else inside & ok
            grids.append(d.view(view))
        z, y, x = grids
        r2 = x * x + y * y + z * z
        inside = inside & (r2 > 0)
        r2 = torch.where(inside, r2, torch.ones_like(r2))
        r = torch.sqrt(r2)
        e = torch.polar(torch.where(inside, 1.0 / (r2 * r), torch.zeros_like(r)), k * r)
        f = torch.complex(-1.0 / r2, k / r)
        del r, inside
        self.spec = []
        for a, b in ((x, x), (x, y), (x, z), (y, y), (y, z), (z, z)):
            d = r2 if a is b else 0.0
            self.spec.append(torch.fft.fftn(e * (k * k * (a * b - d) + f * (3 * a * b - d))))
        del e, f, r2
        if with_target:
            mask = _mask(case, DEV)
            self.sites = mask.reshape(-1).nonzero().reshape(-1)
            self.mat = _materials(case, DEV).reshape(-1)[self.sites].long()
            self.ainv = _alpha_inverse(case, k)[self.mat]

    def product(self, p):
        """A p for p of shape (3, N_d)."""
        hat = []
        for c in range(3):
            v = torch.zeros(math.prod(self.n), dtype=torch.complex128, device=DEV)
            v[self.sites] = p[c]
            hat.append(torch.fft.fftn(v.view(self.n), s=self.L))
        rows, out = ((0, 1, 2), (1, 3, 4), (2, 4, 5)), []
        for c in range(3):
            g = self.spec[rows[c][0]] * hat[0]
            for d in (1, 2):
                g += self.spec[rows[c][d]] * hat[d]
            g = torch.fft.ifftn(g)[: self.n[0], : self.n[1], : self.n[2]].reshape(-1)[self.sites]
            out.append(g + self.ainv * p[c])
        return torch.stack(out)

    def solve(self, b):
        """A x = b by conjugate gradients with the bilinear form (A is complex symmetric), to 1e-12."""
        x, r = torch.zeros_like(b), b.clone()
        q, rho, stop = r.clone(), (r * r).sum(), 1e-12 * float(b.abs().square().sum().sqrt())
        for _ in range(3000):
            v = self.product(q)
            a = rho / (q * v).sum()
            x, r = x + a * q, r - a * v
            if float(r.abs().square().sum().sqrt()) <= stop:
                return x
            new = (r * r).sum()
            q, rho = r + new / rho * q, new
        return None

    def field(self, case, k, khat, e):
        K, J, _ = _shape(case)
        s = self.sites
        x, y, z = (v.to(torch.float64) for v in (s % K, s // K % J, s // (K * J)))
        phase = k * (float(khat[0]) * x + float(khat[1]) * y + float(khat[2]) * z)
        return torch.tensor(e, dtype=torch.complex128, device=DEV)[:, None] * torch.polar(torch.ones_like(phase), phase)

    def cross(self, k, E, P):
        w = -self.ainv.imag - 2.0 / 3.0 * k**3
        ext, ab = (E.conj() * P).imag.sum(), (w * P.abs().square()).sum()
        return [float(4 * math.pi * k * v) for v in (ext, ab, ext - ab)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "setup":
        k = _k(case) * (1.0 + 0.01 * (seed % 16))
        full = _Exact(case, k, with_target=False)
        h = [L // 2 + 1 for L in full.L]
        s = torch.stack([v[: h[0], : h[1], : h[2]].permute(1, 2, 0) for v in full.spec], dim=-1) / math.prod(full.L)
        return {"bits": None, "ranks": None, "spectrum": s}
    k = _k(case)
    # a solve on a large lattice takes minutes this way
    if kind in ("solve", "gradient") and case["nb"] * math.prod(_padded(n) for n in _shape(case)) > 2**25:
        return None
    state = prepare(case, seed)
    full = _Exact(case, k)
    if kind == "product":
        return torch.stack([full.product(p.to(torch.complex128)) for p in state["p"]])
    E = torch.stack([full.field(case, k, kh, e) for kh, e in state["inc"]])
    if kind == "observe":
        return {"E": E, "cross": np.array([full.cross(k, a, b) for a, b in zip(E, state["P"])])}
    P = [full.solve(e) for e in E]
    if any(p is None for p in P):
        return None
    out = {"P": torch.stack(P), "cross": np.array([full.cross(k, a, b) for a, b in zip(E, P)])}
    if kind == "gradient":
        # C_abs = 4 pi k sum w |P|^2, A P = E, w = -Im a - 2/3 k^3: with A mu = w conj(P) and a' = da/d eps,
        # dC/dRe eps = 4 pi k sum_c [-|P|^2 Im a' - 2 Re(mu a' P)], dC/dIm eps = 4 pi k sum_c [-|P|^2 Re a' + 2 Im(mu a' P)]
        w, da = -full.ainv.imag - 2.0 / 3.0 * k**3, _alpha_inverse(case, k, derivative=True)[full.mat]
        mu = full.solve(w * P[0].conj())
        if mu is None:
            return None
        s, a2 = (mu * da * P[0]).sum(0), P[0].abs().square().sum(0)
        grad = 4 * math.pi * k * torch.complex(-a2 * da.imag - 2 * s.real, -a2 * da.real + 2 * s.imag)
        sums = torch.stack([grad[full.mat == q].sum() for q in range(case["nmat"])])
        out.update(grad=grad, sums=sums.cpu().numpy())
    return out
