"""The work a user of this library has it do, as cases that can be timed and compared.

A case is a dict of plain values: ``kind`` names the entry point, the rest its sizes and
options.  ``prepare`` makes what a program holds before the call (gauge field resident on the
device, sources), ``run`` makes the call, ``work`` counts what the call cannot do without, and
``exact`` gives the same outputs from a plain complex128 torch computation.

kind        entry point                              stands for
mdagm       Gauge.mdagm                              the operator of every solve, Mhat^dag Mhat p
hop         Gauge.dslash_eo                          one even-odd hop with its fused axpy and norm
dirac       Gauge.dirac_apply                        D or D^dag on the whole lattice (residuals, heatbath)
solve       Gauge.cg_solve                           one propagator from page-locked host buffers
solve_dev   Gauge.cg_solve_dev                       the same on device buffers
batch       Context.cg_solve_batch                   many sources on two lattices at once
force       Gauge.fermi_force_dev                    U dS/dU of a molecular-dynamics step
multishift  Gauge.cg_multishift_dev                  the shifted solves of a rational approximation
staggered   Gauge.stag_solve_dev                     a staggered propagator
stag_apply  Gauge.stag_apply                         the staggered operator on the whole lattice
hmc         Gauge.hmc_trajectory, Gauge.download     one trajectory and its new links
"""
import math

import numpy as np
import torch

from paper_2409_03030_gb300 import jqcd

PRECS = {"dw": jqcd.PREC_DW, "f32": jqcd.PREC_F32, "f16": jqcd.PREC_F16N, "f64": jqcd.PREC_F64}
MODES = {"dw": jqcd.CG_DW, "f64": jqcd.CG_F64, "mixed_f32": jqcd.CG_MIXED_F32, "mixed_f16": jqcd.CG_MIXED_F16}


def _case(kind, dims, **more):
    c = {"kind": kind, "nx": dims[0], "ny": dims[1], "nz": dims[2], "nt": dims[3], "antiperiodic": True, "eps": 0.3, "kappa": 0.12}
    c.update(more)
    return c


def _dims(c):
    return (c["nx"], c["ny"], c["nz"], c["nt"])


def listed():
    big, mid, sq = (32, 32, 32, 64), (24, 24, 24, 48), (16, 16, 16, 16)
    return [
        # the smallest lattice that is served: launches and latency
        _case("mdagm", (8, 8, 8, 8), name="mdagm_dw_8", prec="dw", norm=True),
        # both parities on a lattice that stays in L2, the adjoint, single precision
        _case("dirac", sq, name="dirac_f32_16", prec="f32", dagger=True),
        # extents that are no powers of two, a ragged last block, periodic time
        _case("mdagm", (20, 18, 14, 26), name="mdagm_dw_ragged", prec="dw", norm=False, antiperiodic=False),
        # the operator at the size the headline solve is quoted on
        _case("mdagm", mid, name="mdagm_dw_24x48", prec="dw", norm=True),
        # the inner operator of the mixed solve at the largest size
        _case("mdagm", big, name="mdagm_f16_32x64", prec="f16", norm=True, eps=0.4, kappa=0.122),
        # a solve in double-word arithmetic inside a device-resident program
        _case("solve_dev", sq, name="solve_dw_16", mode="dw", tol=1e-10, eo=True),
        # the largest propagator, host to host
        _case("solve", big, name="solve_f16_32x64", mode="mixed_f16", tol=1e-10, eo=True, eps=0.4, kappa=0.122),
        # twelve point sources and twelve Gaussian ones on lattices of uneven size
        _case("batch", mid, name="batch_24", mode="mixed_f16", tol=1e-10, count=24, small=16),
        # fermion force, two-flavour action
        _case("force", mid, name="force_24x48"),
        # eight poles of a rational approximation
        _case("multishift", mid, name="multishift_24x48", tol=1e-10, shifts=8),
        # staggered propagator at a light mass
        _case("staggered", mid, name="staggered_24x48", tol=1e-10, mass=0.05),
        # one trajectory with fermions
        _case("hmc", sq, name="hmc_16", mode="dw", tol=1e-10, steps=10, beta=5.5, fermions=True),
    ]


def _draw_dims(rng, low, high):
    """Even extents; the volume's logarithm is uniform between low's and high's."""
    want = math.exp(rng.uniform(math.log(low), math.log(high)))
    while True:
        side = want ** 0.25
        d = [max(2, 2 * round(side * rng.uniform(0.6, 1.6) / 2)) for _ in range(3)]
        t = max(2, 2 * round(want / (d[0] * d[1] * d[2]) / 2))
        v = d[0] * d[1] * d[2] * t
        if t <= 4 * max(d) and 0.8 * low <= v <= high:
            return (d[0], d[1], d[2], t)


def draw(rng):
    big, mid = 32 ** 3 * 64, 24 ** 3 * 48
    kind = rng.choice(["mdagm", "mdagm", "hop", "dirac", "solve", "solve", "solve_dev", "batch", "force", "multishift",
                       "staggered", "stag_apply", "hmc"])
    more = {"antiperiodic": rng.random() < 0.75, "eps": round(rng.uniform(0.2, 0.4), 3), "kappa": round(rng.uniform(0.10, 0.122), 4)}
    tol = rng.choice([1e-8, 1e-10, 1e-12])
    if kind in ("mdagm", "hop", "dirac"):
        more["prec"] = rng.choice(["dw", "dw", "dw", "f32", "f16", "f64"])
        dims = _draw_dims(rng, 4 ** 4, mid if more["prec"] == "f64" else big)
        if kind == "mdagm":
            more["norm"] = rng.random() < 0.5
        else:
            more["dagger"] = rng.random() < 0.5
        if kind == "hop":
            more.update(parity=rng.randrange(2), axpy=rng.random() < 0.5, norm=rng.random() < 0.5)
    elif kind in ("solve", "solve_dev"):
        more["mode"] = rng.choice(["dw", "mixed_f16", "mixed_f16", "mixed_f32", "f64"])
        more["eo"] = True if more["mode"].startswith("mixed") else rng.random() < 0.75
        more["tol"] = tol
        dims = _draw_dims(rng, 4 ** 4, {"dw": mid // 2, "f64": 16 ** 4}.get(more["mode"], big // 2))
    elif kind == "batch":
        more.update(mode=rng.choice(["mixed_f16", "mixed_f16", "mixed_f32"]), tol=tol, count=2 * rng.randint(1, 10), small=2 * rng.randint(2, 7))
        dims = _draw_dims(rng, 8 ** 4, mid // 2)
    elif kind == "force":
        dims = _draw_dims(rng, 4 ** 4, mid)
    elif kind == "multishift":
        more.update(tol=rng.choice([1e-8, 1e-10]), shifts=rng.randint(1, 12))
        dims = _draw_dims(rng, 4 ** 4, mid // 2)
    elif kind == "staggered":
        more.update(tol=rng.choice([1e-8, 1e-10]), mass=round(rng.uniform(0.05, 0.5), 3))
        dims = _draw_dims(rng, 4 ** 4, mid)
    elif kind == "stag_apply":
        more.update(mass=round(rng.uniform(0.05, 0.5), 3), dagger=rng.random() < 0.5)
        dims = _draw_dims(rng, 4 ** 4, mid)
    else:
        more.update(mode=rng.choice(["dw", "mixed_f16"]), tol=1e-10, steps=rng.randint(2, 10), beta=round(rng.uniform(5.3, 6.0), 2),
                    fermions=rng.random() < 0.75)
        dims = _draw_dims(rng, 4 ** 4, 16 ** 4)
    return _case(kind, dims, **more)


# ---- inputs --------------------------------------------------------------------
# Canonical orders: spinors [spin, t, z, y, x, colour], links [mu, t, z, y, x, b, a] (element
# (a, b) of U_mu(x)), staggered fields [t, z, y, x, colour], complex128.

def _normal(gen, *shape):
    """Complex normals, re and im ~ N(0, 1/2)."""
    return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, device="cuda", dtype=torch.float64) * math.sqrt(0.5))


def _mul3(a, b):
    return sum(a[..., :, k, None] * b[..., None, k, :] for k in range(3))


def _links(gen, dims, eps):
    """exp(i eps H), H traceless Hermitian Gaussian: [mu, t, z, y, x, a, b]."""
    nx, ny, nz, nt = dims
    out = torch.empty(4, nt, nz, ny, nx, 3, 3, dtype=torch.complex128, device="cuda")
    one = torch.eye(3, dtype=torch.complex128, device="cuda")
    for mu in range(4):
        a = _normal(gen, nt, nz, ny, nx, 3, 3)
        h = 0.5 * (a + a.mH)
        h = h - one * (h.diagonal(dim1=-2, dim2=-1).sum(-1) / 3)[..., None, None]
        x = (1j * eps / 16) * h
        u = one + x / 12
        for n in range(11, 0, -1):
            u = one + _mul3(x, u) / n
        for _ in range(4):
            u = _mul3(u, u)
        out[mu] = u
    return out


def _host(t):
    """A page-locked host copy, as an array."""
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h.numpy()


def _point(dims, spin, colour):
    nx, ny, nz, nt = dims
    b = torch.zeros(4, nt, nz, ny, nx, 3, dtype=torch.complex128, device="cuda")
    b[spin, 0, 0, 0, 0, colour] = 1
    return b


def _spinor(gen, dims):
    nx, ny, nz, nt = dims
    return _normal(gen, 4, nt, nz, ny, nx, 3)


def _inputs(c, seed):
    """Links, and the vectors of the case, on the device."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    dims, kind = _dims(c), c["kind"]
    U = _links(gen, dims, c["eps"])
    if kind == "batch":
        half, small = c["count"] // 2, (c["small"],) * 4
        U2 = _links(gen, small, c["eps"])
        first = [_point(dims, (i // 3) % 4, i % 3) for i in range(half)]
        return U, U2, first + [_spinor(gen, small) for _ in range(half)]
    if kind in ("staggered", "stag_apply"):
        return U, [_normal(gen, dims[3], dims[2], dims[1], dims[0], 3)]
    return U, [_spinor(gen, dims) for _ in range(2 if kind in ("force", "hop") else 1)]


_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = jqcd.Context(0)
    return _ctx


class State:
    """What a program holds between calls; its gauge fields leave the device with it."""

    def __init__(self, case):
        self.case, self.gauges, self.calls = case, [], 0

    def upload(self, dims, U, antiperiodic):
        g = _context().gauge_upload(dims, _host(U.transpose(-1, -2)), antiperiodic)
        self.gauges.append(g)
        return g

    def __del__(self):
        for g in self.gauges:
            g.free()


def prepare(case, seed):
    c, dims, kind, anti = case, _dims(case), case["kind"], case["antiperiodic"]
    s = State(case)
    if kind == "batch":
        U, U2, bs = _inputs(c, seed)
        big, small = s.upload(dims, U, anti), s.upload((c["small"],) * 4, U2, anti)
        half = c["count"] // 2
        s.fields = [big] * half + [small] * half
        s.b = [_host(b) for b in bs]
        s.x = [_host(torch.zeros_like(b)) for b in bs]
        return s
    if kind == "hmc":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        nx, ny, nz, nt = dims
        g = s.upload(dims, _links(gen, dims, c["eps"]), anti)
        # the random numbers of four trajectories, used in turn
        s.noise = [(torch.randn(4, nt, nz, ny, nx, 8, generator=gen, device="cuda", dtype=torch.float64).cpu().numpy(),
                    _spinor(gen, dims).cpu().numpy() if c["fermions"] else None) for _ in range(4)]
        s.g = g
        return s
    U, vs = _inputs(c, seed)
    g = s.g = s.upload(dims, U, anti)
    del U
    if kind in ("staggered", "stag_apply"):
        s.b = g.stag_pack(vs[0].cpu().numpy())
        s.x = (g.stag_empty(), g.stag_empty())
    elif kind == "solve":
        s.b, s.x = _host(vs[0]), _host(torch.zeros_like(vs[0]))
    elif kind == "force":
        s.X, s.Y = (g.pack(v.cpu().numpy(), jqcd.PREC_DW) for v in vs)
        s.out = torch.empty(g.linkfield_bytes(), dtype=torch.uint8, device="cuda")
    elif kind == "multishift":
        s.b, _ = g.pack(vs[0].cpu().numpy(), jqcd.PREC_DW)
        s.x = [g.empty(jqcd.PREC_DW) for _ in range(c["shifts"])]
    else:
        prec = PRECS[c.get("prec", "dw")]
        s.v = [g.pack(v.cpu().numpy(), prec) for v in vs]
        s.out = (g.empty(prec), g.empty(prec))
        s.norm2 = torch.zeros(1, dtype=torch.float64, device="cuda") if c.get("norm") else None
    torch.cuda.synchronize()
    return s


def _shifts(n):
    """n poles spread geometrically over 1e-4 .. 0.3, the larger residues last."""
    return [1e-4 * 3000.0 ** (i / max(1, n - 1)) for i in range(n)]


def _values(buf, prec, vh):
    """The numbers of a device spinor buffer in its documented layout."""
    if prec == "f64":
        return buf.view(torch.float64)
    if prec == "f16":
        return [buf[: 48 * vh].view(torch.float16), buf[48 * vh:].view(torch.float32)]
    return buf.view(torch.float32)


def run(state):
    s, c = state, state.case
    kind, dims = c["kind"], _dims(c)
    vh = dims[0] * dims[1] * dims[2] * dims[3] // 2
    if kind in ("mdagm", "hop", "dirac"):
        prec = PRECS[c["prec"]]
        even, odd = s.v[0]
        if kind == "mdagm":
            s.g.mdagm(prec, c["kappa"], even, s.out[0], norm2=s.norm2)
        elif kind == "dirac":
            s.g.dirac_apply(prec, c["kappa"], c["dagger"], even, odd, s.out[0], s.out[1])
            return [_values(o, c["prec"], vh) for o in s.out]
        else:
            p = c["parity"]
            x = s.v[1][p] if c["axpy"] else None
            s.g.dslash_eo(prec, p, c["dagger"], s.v[0][1 - p], x, s.out[0], 1.0, -c["kappa"], norm2=s.norm2)
        return [_values(s.out[0], c["prec"], vh)] + ([] if s.norm2 is None else [s.norm2])
    if kind == "solve":
        x, info, _ = s.g.cg_solve(s.b, c["kappa"], tol=c["tol"], eo=c["eo"], mode=MODES[c["mode"]], out=s.x)
        return [x]
    if kind == "solve_dev":
        s.g.cg_solve_dev(s.v[0][0], s.v[0][1], s.out[0], s.out[1], c["kappa"], tol=c["tol"], eo=c["eo"], mode=MODES[c["mode"]])
        return [o.view(torch.float32) for o in s.out]
    if kind == "batch":
        n = c["count"]
        xs, infos, _ = _context().cg_solve_batch(s.fields, s.b, [c["kappa"]] * n, [c["tol"]] * n, mode=MODES[c["mode"]], out=s.x)
        return list(xs)
    if kind == "force":
        s.g.fermi_force_dev(c["kappa"], *s.X, *s.Y, s.out)
        return [s.out.view(torch.float32)]
    if kind == "multishift":
        s.g.cg_multishift_dev(s.b, s.x, c["kappa"], _shifts(c["shifts"]), tol=c["tol"])
        return [x.view(torch.float32) for x in s.x]
    if kind == "staggered":
        s.g.stag_solve_dev(*s.b, *s.x, c["mass"], tol=c["tol"])
        return [x.view(torch.float32) for x in s.x]
    if kind == "stag_apply":
        s.g.stag_apply(c["mass"], c["dagger"], *s.b, *s.x)
        return [x.view(torch.float32) for x in s.x]
    normals, xi = s.noise[s.calls % len(s.noise)]
    s.calls += 1
    info, _ = s.g.hmc_trajectory(normals, xi, 0.0, c["beta"], kappa=c["kappa"], tau=0.1 * c["steps"], n_md=c["steps"], tol=c["tol"],
                                 mode=MODES[c["mode"]])
    return [s.g.download(), info["H_new"], info["plaquette"]]


# ---- what a call cannot do without ----------------------------------------------
# Bytes per site of one parity: a spinor, and the eight links of a hop.  An operator that is
# applied several times, each time to the result of the whole lattice before, reads its links
# each time.

_SPINOR = {"dw": 192, "f64": 192, "f32": 96, "f16": 52}
_LINKS = {"dw": 1152, "f64": 1152, "f32": 384, "f16": 384}


def _iterations(c):
    """About the CG iterations to tol (a little under 66 at 1e-10, kappa 0.12)."""
    k = c["kappa"]
    rate = 5.6 if c.get("eo", True) else 11.0
    return max(4.0, rate * -math.log10(c["tol"]) * (0.12 / (0.24 - k)) ** 2 * 1.1)


def _hop_bytes(prec, axpy):
    return _LINKS[prec] + _SPINOR[prec] * (3 if axpy else 2)


def work(case):
    c, dims, kind = case, _dims(case), case["kind"]
    vh = dims[0] * dims[1] * dims[2] * dims[3] // 2
    hop_flops = 1320.0 * vh
    if kind in ("hop", "mdagm", "dirac"):
        p = c["prec"]
        if kind == "hop":
            return {"bytes": vh * _hop_bytes(p, c["axpy"]), "flops": hop_flops}
        if kind == "dirac":
            return {"bytes": 2 * vh * _hop_bytes(p, True), "flops": 2 * hop_flops}
        return {"bytes": 2 * vh * (_hop_bytes(p, False) + _hop_bytes(p, True)), "flops": 4 * hop_flops}

    def cg(vh, mode, tol):
        # four hops, and x, r, p updated: each read and written
        p = {"dw": "dw", "f64": "f64", "mixed_f32": "f32", "mixed_f16": "f16"}[mode]
        vec = 6 * _SPINOR[p] if p in ("dw", "f64") else 4 * 96 + 2 * _SPINOR[p]
        n = _iterations(dict(c, tol=tol))
        scale = 1 if c.get("eo", True) else 2
        return n * scale * vh * (2 * _hop_bytes(p, False) + 2 * _hop_bytes(p, True) + vec), n * scale * 4 * 1320.0 * vh

    if kind in ("solve", "solve_dev"):
        b, f = cg(vh, c["mode"], c["tol"])
        return {"bytes": b + 2 * 384 * vh, "flops": f}
    if kind == "batch":
        half, sh = c["count"] // 2, c["small"] ** 4 // 2
        p = "f16" if c["mode"] == "mixed_f16" else "f32"
        n = _iterations(c)
        # the links of a hop once for all sources on the field
        per = 4 * (half * (2.5 * _SPINOR[p]) + _LINKS[p]) + half * (4 * 96 + 2 * _SPINOR[p])
        return {"bytes": n * (vh + sh) * per, "flops": n * half * (vh + sh) * 4 * 1320.0}
    if kind == "force":
        # X, Y once, four links and four results a site of the whole lattice
        return {"bytes": 2 * vh * 1536, "flops": 2 * vh * 4 * (2 * 9 * 2 * 8 + 2 * 48 + 216.0)}
    if kind == "multishift":
        n = _iterations(c)
        return {"bytes": n * vh * (2 * _hop_bytes("dw", False) + 2 * _hop_bytes("dw", True) + 4 * 192) + vh * 192 * (c["shifts"] + 1),
                "flops": n * vh * (4 * 1320.0 + c["shifts"] * 24 * 6)}
    if kind in ("staggered", "stag_apply"):
        hop = 1152 + 3 * 48
        if kind == "stag_apply":
            return {"bytes": 2 * vh * hop, "flops": 2 * vh * 570.0}
        n = 14.0 * -math.log10(c["tol"]) / math.sqrt(c["mass"]) * 0.35
        return {"bytes": n * vh * (2 * hop + 6 * 48), "flops": n * vh * 2 * 570.0}
    # hmc: per step the links twice (read, exponential, written in FP64 and both copies), the
    # staple force, and two solves
    links = 2 * vh * 4 * 144
    b, f = c["steps"] * 6 * links, c["steps"] * 2 * vh * 4 * (6 * 2 * 216 + 216 + 2 * 400.0)
    if c["fermions"]:
        sb, sf = cg(vh, c["mode"], c["tol"])
        b, f = b + 2 * (c["steps"] + 1) * sb, f + 2 * (c["steps"] + 1) * sf
    return {"bytes": b, "flops": f}


# ---- the same in 64 bits, by plain torch -----------------------------------------
# gamma_mu psi in the DeGrand-Rossi basis: spin source and phase of each row.
_GAMMA = [([3, 2, 1, 0], [1j, 1j, -1j, -1j]), ([3, 2, 1, 0], [-1, 1, 1, -1]), ([2, 3, 0, 1], [1j, -1j, -1j, 1j]), ([2, 3, 0, 1], [1, 1, 1, 1])]
_AXIS = [4, 3, 2, 1]  # of x, y, z, t in [mu or spin, t, z, y, x, ...]


def _gamma(psi, mu):
    src, ph = _GAMMA[mu]
    return psi[src] * torch.tensor(ph, dtype=psi.dtype, device=psi.device).view(4, 1, 1, 1, 1, 1)


def _shift(f, mu, step, anti):
    """f(x + step mu), step +-1, with the sign of the time boundary."""
    g = torch.roll(f, -step, _AXIS[mu])
    if mu == 3 and anti:
        g.select(1, -1 if step > 0 else 0).mul_(-1)
    return g


def _apply(U, psi, adjoint=False):
    """U psi (or U^dag psi) for psi [spin, ..., colour]."""
    W = U.mH if adjoint else U
    return sum(W[None, ..., :, k] * psi[..., k, None] for k in range(3))


def _hop_exact(U, psi, anti, dagger=False):
    out = torch.zeros_like(psi)
    for mu in range(4):
        s = 1 if dagger else -1
        f = _apply(U[mu], _shift(psi, mu, 1, anti))
        out += f + s * _gamma(f, mu)
        b = _shift(_apply(U[mu], psi, True), mu, -1, anti)
        out += b - s * _gamma(b, mu)
    return out


def _parity(dims, device="cuda"):
    nx, ny, nz, nt = dims
    r = [torch.arange(n, device=device) for n in (nt, nz, ny, nx)]
    return (r[0][:, None, None, None] + r[1][:, None, None] + r[2][:, None] + r[3]) % 2


def _chunks(psi, parity, p):
    """[component, site of parity p] of psi [spin, t, z, y, x, colour] (or a staggered field, or links)."""
    v = psi.movedim(-1, 1).flatten(2) if psi.dim() == 6 else psi.movedim(-1, 0).flatten(1)[None]
    return v.flatten(0, 1)[:, (parity == p).flatten()]


def _pairs(v):
    """The (re.hi, im.hi, re.lo, im.lo) floats of complex128 chunks."""
    r = torch.view_as_real(v.contiguous())
    h = r.float()
    return torch.cat([h, (r - h.double()).float()], -1).reshape(-1)


def _device_form(v, prec):
    if prec == "dw":
        return _pairs(v)
    r = torch.view_as_real(v.contiguous())  # [12, vh, 2]
    if prec == "f64":
        return r.reshape(-1)
    vh = r.shape[1]
    if prec == "f32":
        return r.reshape(6, 2, vh, 2).transpose(1, 2).reshape(-1)
    n = r.abs().amax((0, 2))
    return [(r / n[None, :, None]).reshape(3, 4, vh, 2).transpose(1, 2).reshape(-1), n]


def _cg(A, b, tol=3e-14, most=6000):
    x, r, p = torch.zeros_like(b), b.clone(), b.clone()
    rr = torch.view_as_real(r).square().sum()
    stop = float(rr) * tol * tol
    for i in range(most):
        q = A(p)
        a = rr / (torch.view_as_real(p) * torch.view_as_real(q)).sum()
        x += a * p
        r -= a * q
        new = torch.view_as_real(r).square().sum()
        p = r + (new / rr) * p
        rr = new
        if i % 10 == 9 and float(rr) <= stop:
            break
    return x


def _solve_exact(U, b, kappa, anti):
    D = lambda v, dag: v - kappa * _hop_exact(U, v, anti, dag)  # noqa: E731
    x = _cg(lambda v: D(D(v, False), True), D(b, True))
    r = b - D(x, False)
    return x + _cg(lambda v: D(D(v, False), True), D(r, True), 1e-4)


def _stag_exact(U, psi, dims, anti):
    """D_hop psi of a staggered field [t, z, y, x, colour]."""
    nx, ny, nz, nt = dims
    x, y, z = (torch.arange(n, device="cuda") for n in (nx, ny, nz))
    eta = [torch.ones(1, 1, 1, 1, device="cuda"), 1 - 2.0 * (x % 2).view(1, 1, 1, nx), 1 - 2.0 * ((x + y[:, None]) % 2).view(1, 1, ny, nx),
           1 - 2.0 * ((x + y[:, None] + z[:, None, None]) % 2).view(1, nz, ny, nx)]
    out = torch.zeros_like(psi)
    for mu in range(4):
        f = _apply(U[mu], _shift(psi[None], mu, 1, anti))
        b = _shift(_apply(U[mu], psi[None], True), mu, -1, anti)
        out += 0.5 * eta[mu][..., None] * (f - b)[0]
    return out


def exact(case, seed):
    c, dims, kind, anti = case, _dims(case), case["kind"], case["antiperiodic"]
    k, vol = c["kappa"], dims[0] * dims[1] * dims[2] * dims[3]
    if kind == "hmc":
        return None
    par = _parity(dims)
    even = (par == 0)[None, ..., None]
    if kind == "batch":
        U, U2, bs = _inputs(c, seed)
        half, out = c["count"] // 2, [None] * c["count"]
        for i in {0, half // 2, half, c["count"] - 1}:  # the others alike
            out[i] = _solve_exact(U if i < half else U2, bs[i], k, anti).cpu().numpy()
        return out
    U, vs = _inputs(c, seed)
    psi = vs[0]
    if kind == "hop":
        p = c["parity"]
        keep = even if p == 0 else ~even
        h = -k * _hop_exact(U, torch.where(keep, 0, psi), anti, c["dagger"])
        out = torch.where(keep, h + vs[1] if c["axpy"] else h, 0)
        return [_device_form(_chunks(out, par, p), c["prec"])] + ([torch.view_as_real(out).square().sum()[None]] if c["norm"] else [])
    if kind == "dirac":
        out = psi - k * _hop_exact(U, psi, anti, c["dagger"])
        return [_device_form(_chunks(out, par, p), c["prec"]) for p in (0, 1)]
    H = lambda v, dag: torch.where(even, _hop_exact(U, _hop_exact(U, v, anti, dag), anti, dag), 0)  # noqa: E731
    M = lambda v, dag: v - k * k * H(v, dag)  # noqa: E731
    if kind == "mdagm":
        w = M(torch.where(even, psi, 0), False)
        return [_device_form(_chunks(M(w, True), par, 0), c["prec"])] + ([torch.view_as_real(w).square().sum()[None]] if c["norm"] else [])
    if kind in ("solve", "solve_dev"):
        x = _solve_exact(U, psi, k, anti)
        return [x.cpu().numpy()] if kind == "solve" else [_pairs(_chunks(x, par, p)) for p in (0, 1)]
    if kind == "multishift":
        if vol * c["shifts"] > 3 * 24 ** 3 * 48:
            # the first, the middle and the last pole
            todo = {0, c["shifts"] // 2, c["shifts"] - 1}
        else:
            todo = set(range(c["shifts"]))
        b = torch.where(even, psi, 0)
        return [_pairs(_chunks(_cg(lambda v: M(M(v, False), True) + sg * v, b), par, 0)) if i in todo else None
                for i, sg in enumerate(_shifts(c["shifts"]))]
    if kind == "stag_apply":
        h = _stag_exact(U, psi, dims, anti)
        out = c["mass"] * psi + (-h if c["dagger"] else h)
        return [_pairs(_chunks(out, par, p)) for p in (0, 1)]
    if kind == "staggered":
        m = c["mass"]
        h = lambda v: _stag_exact(U, v, dims, anti)  # noqa: E731
        x = _cg(lambda v: m * m * v - h(h(v)), m * psi - h(psi))
        return [_pairs(_chunks(x, par, p)) for p in (0, 1)]
    # force: 2 kappa s U (A + B^dag)
    X, Y = vs
    parts = [[], []]
    for mu in range(4):
        xf, yf = (_shift(f, mu, 1, anti) for f in (X, Y))
        a, b = xf - _gamma(xf, mu), X + _gamma(X, mu)
        A = sum(a[s][..., :, None] * Y[s].conj()[..., None, :] for s in range(4))
        B = sum(b[s][..., :, None] * yf[s].conj()[..., None, :] for s in range(4))
        G = 2 * k * _mul3(U[mu], A + B.mH)
        for p in (0, 1):
            parts[p].append(G.flatten(-2).movedim(-1, 0).flatten(1)[:, (par == p).flatten()])
    return [_pairs(torch.cat(parts[0] + parts[1]))]
