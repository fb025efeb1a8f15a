"""The calls whose speed counts, each one pass through the library's public functions.

A program of this library loads a gauge configuration, applies the stencil,
converts fields between FP64 and the storage formats, and above all solves:
one system, twelve shifted systems, a batch of right-hand sides, the full
lattice.  The lattices are those of the library's own configurations and tests
(8^4, 16^4, 24^3x48, 32^3x64 and ragged ones with extents that are no powers of
two); links are SU(3) matrices exp(i 0.3 H) near the identity with staggered
phases, fat ones scaled by 0.8, sources Gaussian.

listed() names the cases, draw() gives more of the same ranges, prepare() makes
the inputs on the GPU, run() is one pass, exact() the same result in 64 bits
from plain torch operations, work() the compulsory bytes and flops of a pass.
"""
import math

import torch

from paper_2302_09224_gb300 import hisq

EPS = 0.3         # links exp(i EPS H)
FAT_SCALE = 0.8   # fat links: scaled SU(3)
LAMBDA_MAX = 20.0  # about the largest eigenvalue of -D_eo D_oe for such links
EXACT_SITES = 16 * 16 * 16 * 32  # largest lattice whose solves exact() repeats in 64 bits
FLOPS_SITE = 1146  # one stencil pass, per output site


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: one parity of the operator inside a caller's own iteration, 20-bit fields
        _stencil("dslash_int20_8x8x8x8", (8, 8, 8, 8), "int20", 12, parity=0, a=0.0, antiperiodic=False),
        # a ragged lattice, antiperiodic in t, the full operator 2m - D in the 16-bit format
        _stencil("dslash_half_full_ragged", (6, 10, 14, 22), "half", 12, parity=2, a=0.1, antiperiodic=True),
        # a true residual in FP64: what decides convergence in every solver
        _stencil("dslash_f64_16x16x16x32", (16, 16, 16, 32), "f64", 18, parity=0, a=0.04, antiperiodic=False),
        # the production lattice, full operator, 20-bit fields: bandwidth
        _stencil("dslash_int20_full_32x32x32x64", (32, 32, 32, 64), "int20", 12, parity=2, a=0.02,
                 antiperiodic=False),
        # storage of propagators: FP64 fields to 20-bit records and back, a site count that no block divides
        dict(name="codec_int20", kind="codec", fmt="int20", n=24 * 24 * 24 * 48 + 37),
        # a new configuration (one molecular-dynamics step): load, first use in the 20-bit triplet, release
        _case("load_and_apply_16x16x16x32", "load", (16, 16, 16, 32), fmt="int20", recon=12),
        # one solve on a small lattice: launches and latency
        _solve("cg_int20_8x8x8x8", "cg", (8, 8, 8, 8), 0.1, 1e-10, "int20", 12),
        # the library's headline configuration: one even/odd solve with 20-bit sloppy fields
        _solve("cg_int20_32x32x32x64", "cg", (32, 32, 32, 64), 0.01, 1e-10, "int20", 12),
        # the full-lattice system by even/odd reduction, 16-bit sloppy fields
        _solve("full_half_16x16x16x16", "full", (16, 16, 16, 16), 0.05, 1e-11, "half", 12),
        # RHMC's rational approximation: twelve shifts, 30-bit stage with FP64-class arithmetic, 20-bit refinement
        _solve("multishift_12_16x16x16x32", "multishift", (16, 16, 16, 32), 0.05, 1e-11, "int30", 18, count=12),
        # a propagator's sources (colours by spin tastes) solved together
        _solve("batched_16_24x24x24x48", "batched", (24, 24, 24, 48), 0.05, 1e-11, "int20", 12, count=16),
        # BiCGStab(4) on the unpreconditioned operator
        _solve("bicgstab4_int20_16x16x16x32", "bicgstab", (16, 16, 16, 32), 0.05, 1e-11, "int20", 12),
    ]


def draw(rng):
    """One more case of the listed ones' kinds, its lattice spread over the same volumes."""
    kind = rng.choice(["dslash", "dslash", "dslash", "codec", "load", "cg", "cg", "full", "multishift", "batched",
                       "bicgstab"])
    if kind == "codec":
        n = int(2048 * (32 * 32 * 32 * 32 / 2048.0) ** rng.random()) | 1
        return dict(kind="codec", fmt=rng.choice(["int20", "half", "int30", "f32", "int14"]), n=n)
    if kind == "dslash":
        fmt, recon = rng.choice([("int20", 12), ("half", 12), ("f32", 12), ("f64", 18), ("int30", 18), ("int14", 12),
                                 ("int20", 18)])
        return _stencil(None, _dims(rng, 8 ** 4, 32 ** 3 * 64), fmt, recon, parity=rng.randrange(3),
                        a=rng.choice([0.0, round(rng.uniform(0.02, 0.3), 3)]), antiperiodic=rng.random() < 0.5)
    if kind == "load":
        fmt, recon = rng.choice([("int20", 12), ("half", 12), ("f32", 12), ("int30", 18)])
        return _case(None, kind, _dims(rng, 8 ** 4, 24 ** 3 * 48), fmt=fmt, recon=recon)
    mass = round(0.05 * 4.0 ** rng.random(), 4)
    fmt, recon = rng.choice([("int20", 12), ("half", 12), ("f32", 12)])
    if kind == "multishift":
        fmt, recon = rng.choice([("int30", 18), ("f32", 12), ("int20", 12)])
        return _solve(None, kind, _dims(rng, 8 ** 4, 16 ** 3 * 32), mass, 1e-11, fmt, recon,
                      count=rng.randrange(8, 13))
    if kind == "batched":
        return _solve(None, kind, _dims(rng, 8 ** 4, 16 ** 3 * 32), mass, 1e-11, fmt, recon,
                      count=rng.choice([2, 4, 8, 12, 16]))
    return _solve(None, kind, _dims(rng, 8 ** 4, 24 ** 3 * 48 if kind == "cg" else 16 ** 3 * 32), mass, 1e-11, fmt,
                  recon)


def _case(name, kind, dims, **more):
    c = {"name": name} if name else {}
    c.update(kind=kind, x=dims[0], y=dims[1], z=dims[2], t=dims[3], **more)
    return c


def _stencil(name, dims, fmt, recon, parity, a, antiperiodic):
    return _case(name, "dslash", dims, fmt=fmt, recon=recon, parity=parity, a=a, antiperiodic=antiperiodic)


def _solve(name, kind, dims, mass, tol, fmt, recon, count=1):
    return _case(name, kind, dims, mass=mass, tol=tol, fmt=fmt, recon=recon, count=count)


def _dims(rng, lo, hi):
    """Even extents whose volume lies between lo and hi, spread over its logarithm."""
    v = lo * (hi / lo) ** rng.random()
    side = v ** 0.25
    d = [max(4, 2 * round(side * rng.uniform(0.75, 1.1) / 2)) for _ in range(3)]
    t = 2 * round(v / (d[0] * d[1] * d[2]) / 2)
    while d[0] * d[1] * d[2] * t > hi and t > 4:
        t -= 2
    return d[0], d[1], d[2], max(4, t)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
_CTX = None


def _context():
    """The program's one context: it keeps the stream and the buffers of every call."""
    global _CTX
    if _CTX is None:
        _CTX = hisq.hisq_create(0)
    return _CTX


class Gauge:
    """A loaded configuration, released with its last reference."""

    def __init__(self, dims, fat, lng, flags):
        self.ctx = _context()
        self.handle = hisq.hisq_load_gauge(self.ctx, dims, fat, lng, flags)

    def __del__(self):
        hisq.hisq_free_gauge(self.ctx, self.handle)


def _lattice(case):
    return case["x"], case["y"], case["z"], case["t"]


def _sites(case):
    return case["x"] * case["y"] * case["z"] * case["t"]


def _signs(dims, hop, antiperiodic, dev):
    """Staggered phase times boundary sign of every link, [mu][t][z][y][x]."""
    lx, ly, lz, lt = dims
    c = torch.meshgrid(*(torch.arange(n, device=dev) for n in (lt, lz, ly, lx)), indexing="ij")
    t, z, y, x = c
    s = [1 - 2 * (p % 2) for p in (torch.zeros_like(x), x, x + y, x + y + z)]
    if antiperiodic:
        s[3] = torch.where(t >= lt - hop, -s[3], s[3])
    return torch.stack(s).to(torch.float64)


def _links(dims, hop, antiperiodic, scale, gen, dev):
    """One link field, float64 [mu][t][z][y][x][3][3][2]: scale * sign * SU(3) near the identity."""
    lx, ly, lz, lt = dims
    n = 4 * lx * ly * lz * lt
    out = torch.empty((n, 3, 3, 2), dtype=torch.float64, device=dev)
    sign = _signs(dims, hop, antiperiodic, dev).reshape(-1) * scale
    step = 1 << 21
    for i in range(0, n, step):
        m = min(step, n - i)
        g = torch.randn((m, 3, 3, 2), dtype=torch.float32, device=dev, generator=gen)
        g = torch.view_as_complex(g)
        h = 0.5 * (g + g.conj().transpose(1, 2))
        h = h - (torch.diagonal(h, dim1=1, dim2=2).sum(1) / 3)[:, None, None] * torch.eye(3, device=dev)
        a = (1j * EPS / 4) * h
        a2 = _mul(a, a)
        e = torch.eye(3, device=dev) + a + a2 / 2 + _mul(a2, a) / 6 + _mul(a2, a2) / 24
        e = _mul(e, e)
        e = _mul(e, e)[:, :2].to(torch.complex128)
        r0 = e[:, 0] / torch.linalg.vector_norm(e[:, 0], dim=1, keepdim=True)
        r1 = e[:, 1] - (r0.conj() * e[:, 1]).sum(1, keepdim=True) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=1, keepdim=True)
        u = torch.stack([r0, r1, torch.linalg.cross(r0, r1, dim=1).conj()], 1)
        out[i:i + m] = torch.view_as_real(u) * sign[i:i + m, None, None, None]
    return out.reshape(4, lt, lz, ly, lx, 3, 3, 2)


def _mul(a, b):
    return (a[:, :, :, None] * b[:, None, :, :]).sum(2)


def _fields(case, seed):
    """(fat, long) of a case."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(seed)
    anti = bool(case.get("antiperiodic", False))
    dims = _lattice(case)
    return (_links(dims, 1, anti, FAT_SCALE, gen, dev), _links(dims, 3, anti, 1.0, gen, dev)), gen


def _gauss(shape, gen):
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen)


def _shifts(n):
    """Rational-approximation shifts from 1e-4 to 1 and their targets, the case's for the smallest to 1e3 times it."""
    f = [i / max(1, n - 1) for i in range(n)]
    return [1e-4 * 1e4 ** v for v in f], [10.0 ** (1.0 * v) for v in f]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "codec":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        n = case["n"]
        # components of one site share a magnitude, magnitudes differ from site to site
        x = _gauss((n, 3, 2), gen) * torch.exp(2.0 * _gauss((n, 1, 1), gen))
        sf = hisq.SPINOR_FMT[case["fmt"]]
        s = {"ctx": _context(), "case": case, "x": x, "sf": sf, "stream": torch.cuda.Stream(),
             "packed": torch.empty(hisq.hisq_spinor_bytes(sf, n), dtype=torch.uint8, device="cuda"),
             "out": torch.empty_like(x)}
        torch.cuda.synchronize()
        return s
    (fat, lng), gen = _fields(case, seed)
    dims = _lattice(case)
    vh = _sites(case) // 2
    flags = hisq.HISQ_GAUGE_ANTIPERIODIC_T if case.get("antiperiodic", False) else 0
    s = {"ctx": _context(), "case": case, "prec": hisq.prec(case["fmt"], case["recon"])}
    if kind == "load":
        s.update(fat=fat, lng=lng, x=_gauss((vh, 3, 2), gen), out=torch.empty((vh, 3, 2), dtype=torch.float64,
                                                                              device="cuda"))
        torch.cuda.synchronize()
        return s
    torch.cuda.synchronize()  # the library reads the links on its own stream
    s["gauge"] = Gauge(dims, fat, lng, flags)
    full = kind in ("full", "bicgstab") or (kind == "dslash" and case["parity"] == 2)
    n = (2 if full else 1) * vh
    if kind == "dslash":
        s["x"] = _gauss((n, 3, 2), gen)
        s["y"] = _gauss((n, 3, 2), gen) if case["a"] else None
        s["out"] = torch.empty((n, 3, 2), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        return s
    p = hisq.hisq_default_params()
    p.mass, p.tol, p.on_device = case["mass"], case["tol"], 1
    p.sloppy = s["prec"]
    s["params"] = p
    count = case["count"]
    if kind == "multishift":
        sig, rel = _shifts(count)
        s["sigma"], s["tol"] = sig, [case["tol"] * r for r in rel]
        s["b"] = _gauss((vh, 3, 2), gen)
        s["x"] = [torch.empty_like(s["b"]) for _ in range(count)]
    else:
        p.nrhs = count
        s["b"] = _gauss((count, n, 3, 2), gen)
        s["x"] = torch.empty_like(s["b"])
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "codec":
        hisq.hisq_spinor_pack(ctx, s["sf"], case["n"], s["x"], s["packed"], s["stream"])
        hisq.hisq_spinor_unpack(ctx, s["sf"], hisq.HISQ_COMPUTE_F64 if case["fmt"] == "int30" else
                                hisq.HISQ_COMPUTE_F32, case["n"], s["packed"], s["out"], s["stream"])
        return {"packed": s["packed"], "decoded": s["out"]}
    if kind == "load":
        g = hisq.hisq_load_gauge(ctx, _lattice(case), s["fat"], s["lng"], 0)
        hisq.hisq_dslash(ctx, g, s["prec"], 0, 0.0, None, s["x"], s["out"], True)
        scale = [hisq.hisq_gauge_scale(g, 0), hisq.hisq_gauge_scale(g, 1)]
        hisq.hisq_free_gauge(ctx, g)
        return {"out": s["out"], "scale": scale}
    g = s["gauge"].handle
    if kind == "dslash":
        hisq.hisq_dslash(ctx, g, s["prec"], case["parity"], case["a"], s["y"], s["x"], s["out"], True)
        return s["out"]
    if kind == "multishift":
        st, _ = hisq.hisq_multishift_cg(ctx, g, s["params"], s["sigma"], s["tol"], s["b"], s["x"])
    elif kind == "full":
        st, _ = hisq.hisq_solve_full(ctx, g, s["params"], s["b"], s["x"])
    elif kind == "bicgstab":
        st, _ = hisq.hisq_bicgstabl(ctx, g, s["params"], s["b"], s["x"])
    else:
        st, _ = hisq.hisq_cg(ctx, g, s["params"], s["b"], s["x"])
    if st != hisq.HISQ_OK:
        raise RuntimeError("the solve ended with status %d" % st)
    return s["x"]


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
class _Operator:
    """D between the parities of a lattice, complex128, by gathering neighbours."""

    def __init__(self, dims, fat, lng):
        lx, ly, lz, lt = dims
        dev = fat.device
        lex = torch.arange(lx * ly * lz * lt, device=dev)
        x, y, z, t = lex % lx, lex // lx % ly, lex // (lx * ly) % lz, lex // (lx * ly * lz)
        par = (x + y + z + t) % 2
        self.terms = ([], [])
        sites = [lex[par == p] for p in (0, 1)]  # ascending: the checkerboard order
        stride, coord = (1, lx, lx * ly, lx * ly * lz), (x, y, z, t)
        for p in (0, 1):
            s = sites[p]
            for mu in range(4):
                for f, hop in ((fat, 1), (lng, 3)):
                    u = torch.view_as_complex(f[mu].reshape(-1, 3, 3, 2))
                    c = coord[mu][s]
                    up = s + ((c + hop) % dims[mu] - c) * stride[mu]
                    dn = s + ((c - hop) % dims[mu] - c) * stride[mu]
                    self.terms[p].append((u[s], up // 2))
                    self.terms[p].append((-u[dn].conj().transpose(1, 2), dn // 2))

    def d(self, p, v):
        """D v on the sites of parity p, v a complex field [..., Vh, 3] of the other parity."""
        out = torch.zeros_like(v)
        for u, at in self.terms[p]:
            w = v[..., at, :]
            for j in range(3):
                out += u[:, :, j] * w[..., j, None]
        return out

    def mee(self, diag, v):
        return diag * v - self.d(0, self.d(1, v))

    def solve(self, diag, b, tol=1e-14):
        """CG for (diag - D_eo D_oe) x = b, one system."""
        x = torch.zeros_like(b)
        r = b.clone()
        p = r.clone()
        rr = float((r.real ** 2 + r.imag ** 2).sum())
        stop = tol * tol * rr
        for _ in range(20000):
            ap = self.mee(diag, p)
            alpha = rr / float((p.real * ap.real + p.imag * ap.imag).sum())
            x += alpha * p
            r -= alpha * ap
            new = float((r.real ** 2 + r.imag ** 2).sum())
            if new <= stop:
                break
            p = r + (new / rr) * p
            rr = new
        return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "codec":
        s = prepare(case, seed)
        return {"packed": None, "decoded": s["x"]}  # the records are bytes; their values are the input's
    solves = kind not in ("dslash", "load")
    if solves and (_sites(case) > EXACT_SITES or kind == "batched" and _sites(case) * case["count"] > EXACT_SITES):
        return None
    (fat, lng), gen = _fields(case, seed)
    dims, vh = _lattice(case), _sites(case) // 2
    if kind == "load":
        x = torch.view_as_complex(_gauss((vh, 3, 2), gen))
        out = torch.view_as_real(_Operator(dims, fat, lng).d(0, x))
        return {"out": out, "scale": [float(fat.abs().max()), float(lng.abs().max())]}
    op = _Operator(dims, fat, lng)
    if kind == "dslash":
        full = case["parity"] == 2
        n = 2 * vh if full else vh
        x = torch.view_as_complex(_gauss((n, 3, 2), gen))
        y = torch.view_as_complex(_gauss((n, 3, 2), gen)) if case["a"] else None
        if full:
            out = torch.cat([op.d(0, x[vh:]), op.d(1, x[:vh])])
        else:
            out = op.d(case["parity"], x)
        return torch.view_as_real(case["a"] * y - out if case["a"] else out)
    m = case["mass"]
    if kind == "multishift":
        b = torch.view_as_complex(_gauss((vh, 3, 2), gen))
        return [torch.view_as_real(op.solve(4 * m * m + sg, b)) for sg in _shifts(case["count"])[0]]
    full = kind in ("full", "bicgstab")
    b = torch.view_as_complex(_gauss((case["count"], (2 if full else 1) * vh, 3, 2), gen))
    if not full:
        return torch.view_as_real(torch.stack([op.solve(4 * m * m, v) for v in b]))
    be, bo = b[0, :vh], b[0, vh:]
    xe = op.solve(4 * m * m, 2 * m * be - op.d(0, bo))
    xo = (bo - op.d(1, xe)) / (2 * m)
    return torch.view_as_real(torch.cat([xe, xo])[None])


# ---------------------------------------------------------------------------
# compulsory work
# ---------------------------------------------------------------------------
_SITE = {"f64": 48, "f32": 24, "half": 16, "int20": 16, "int30": 24, "int14": 12}
_REAL = {"f64": 8, "f32": 4, "half": 2, "int20": 2, "int30": 4, "int14": 2}


def work(case):
    """Each input once and each output once; a solver's iterations, at the CG's textbook count, each
    stream the stored links once per stencil pass, which no cache holds, and its vectors."""
    kind = case["kind"]
    if kind == "codec":
        return {"bytes": case["n"] * (96.0 + 2 * _SITE[case["fmt"]]), "flops": 0.0}
    vh = _sites(case) // 2
    links = 8.0 * _REAL[case["fmt"]] * (18 + case["recon"])  # of one pass, per output site
    if kind == "load":
        return {"bytes": vh * (2.0 * 4 * 2 * 144 + links + 96), "flops": float(FLOPS_SITE) * vh}
    if kind == "dslash":
        n = vh * (2 if case["parity"] == 2 else 1)
        return {"bytes": n * (links + 96.0 + (48.0 if case["a"] else 0.0)), "flops": float(FLOPS_SITE) * n}
    m2 = 4.0 * case["mass"] ** 2
    systems = case["count"] if kind == "batched" else 1
    passes = 2.0 * math.ceil(0.5 * math.sqrt((LAMBDA_MAX + m2) / m2) * math.log(2.0 / case["tol"]))
    vectors = 4.0 * _SITE[case["fmt"]]  # r, p read and written around the two passes
    return {"bytes": vh * passes * (links + systems * vectors) + 96.0 * vh * case["count"],
            "flops": float(FLOPS_SITE) * vh * passes * systems}
