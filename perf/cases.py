"""Performance cases: the calls a user of this package makes, through its public entry points.

The path is: point-source or noise-source propagators of Dirichlet domains of one resident
gauge field (alone, in uneven batches, through the server, for nested domains), the stencil
powers of the expanded trace, and the mode blocks of the projector cut.  ``listed()`` gives
the sizes the package's own workloads use; ``draw()`` more of the same ranges: odd extents,
wrapped boxes, every storage format, with and without the clover term.

Gauge fields are synthetic: independent SU(3) links near the identity with a mean plaquette
of 0.59, as in the package's own measurements; time is antiperiodic.
"""
import math

import torch

import paper_1601_04587_gb300 as ddp

EPS = 0.50892685          # disorder of the links: mean plaquette 0.59
PREC = {"fp64": ddp.DDP_PREC_FP64, "fp32": ddp.DDP_PREC_MIXED_FP32, "fp16": ddp.DDP_PREC_MIXED_FP16,
        "bf16": ddp.DDP_PREC_MIXED_BF16}
TOL = 1e-10               # relative residual every solve is asked for
EXACT_SITE_COLS = 1_600_000   # larger solves have no 64-bit value here (it takes too long)


# ------------------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest domain of the serving mix: one propagator on a 4^4 block, latency
        _solve("block_4", "16x16x16x16", "4x4x4x4", 0.150, "fp32"),
        # the block of the uneven batch (256 of them tile a 32^4 lattice), here one alone
        _solve("block_8", "16x16x16x16", "8x8x8x8", 0.150, "fp32"),
        # the thin slab of the batch and of the serving mix
        _solve("slab_4x32", "8x32x32x32", "4x32x32x32", 0.150, "fp32"),
        # the O(a)-improved operator on the thinnest slab of the nested series
        _solve("clover_8x24", "16x24x24x24", "8x24x24x24", 0.120, "fp32", csw=1.0),
        # level-1 noise columns of the two-level integration, 16-bit storage
        dict(name="noise_16x24", op="noise", lattice="32x24x24x24", extent="16x24x24x24", kappa=0.137, csw=0.0,
             precision="fp16", ncol=12),
        # an uneven batch in one call: blocks, thin slabs and a ragged box
        dict(name="batch", op="batch", lattice="32x16x16x16", boxes="8x8x8x8*32 4x16x16x16*8 5x7x6x10*4",
             kappa=0.140, precision="fp32"),
        # the server: mixed requests submitted at once, stepped until all are done
        dict(name="serve", op="serve", lattice="32x16x16x16", boxes="4x4x4x4*8 8x8x8x8*8 4x16x16x16*3 8x16x16x16*1",
             kappa=0.140, precision="fp32"),
        # the benchmark step: nested slabs 8, 16, 24 and the whole lattice, propagators and correlators
        dict(name="series_48x24", op="series", lattice="48x24x24x24", slabs="8 16 24 48", kappa=0.137, csw=0.0,
             precision="fp32"),
        # the expanded stochastic trace: eighth power of the hopping term in FP64, and its contraction
        dict(name="expanded_16x24", op="expanded", lattice="32x24x24x24", extent="16x24x24x24", kappa=0.140, p=8,
             ncol=12),
        # modes of the projector cut: one inverse iteration (solve, orthonormalization)
        dict(name="modes_48", op="modes", lattice="16x16x16x16", extent="8x16x16x16", kappa=0.140, precision="fp32",
             m=48, iters=1),
        # pion blocks of the cut with the paper's 120 modes
        dict(name="pion_blocks_120", op="gram", lattice="16x24x24x24", extent="8x24x24x24", m=120),
        # nucleon blocks of the cut, 24 modes
        dict(name="nucleon_blocks_24", op="colourless", lattice="8x24x24x24", extent="4x24x24x24", m=24, form=1),
    ]


def _solve(name, lattice, extent, kappa, precision, csw=0.0, origin="0x0x0x0"):
    return dict(name=name, op="propagator", lattice=lattice, origin=origin, extent=extent, kappa=kappa, csw=csw,
                precision=precision)


def draw(rng):
    op = rng.choice(["propagator"] * 5 + ["noise"] * 2 + ["batch"] * 2 + ["serve", "series", "series", "expanded",
                                                                        "modes", "gram", "colourless"])

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(lo, hi, most=32):
        """Extents of about exp(U(log lo, log hi)) sites, the last one even; any of them odd."""
        n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        s = n ** 0.25
        e = [max(1, min(most, int(round(s * math.exp(rng.uniform(-0.5, 0.5)))))) for _ in range(3)]
        e3 = max(2, min(most, 2 * int(round(s * math.exp(rng.uniform(-0.5, 0.5)) / 2))))
        e[0] = max(1, min(48, int(n / (e[1] * e[2] * e3))))
        return e + [e3]

    def around(e):
        """A lattice the box fits into: some directions unrestricted."""
        return [x if x % 2 == 0 and rng.random() < 0.4 else max(4, 2 * ((x + 2) // 2)) for x in e]

    def kappa_of(n):
        return round(rng.uniform(0.140, 0.150) if n <= 4096 else rng.uniform(0.128, 0.138), 4)

    def fmt(big):
        return rng.choice(["fp32"] * 4 + ["fp16", "bf16"] + ([] if big else ["fp64"]))

    if op == "propagator":
        e = box(64, 150_000)
        n = math.prod(e)
        lat = around(e)
        o = [0 if x == l else rng.randrange(l) for x, l in zip(e, lat)]
        clover = rng.random() < 0.25
        return dict(op=op, lattice=_x(lat), origin=_x(o), extent=_x(e),
                    kappa=round(rng.uniform(0.115, 0.122), 4) if clover else kappa_of(n), csw=1.0 if clover else 0.0,
                    precision=fmt(n > 20_000))
    if op == "noise":
        e = box(256, 200_000)
        n = math.prod(e)
        return dict(op=op, lattice=_x(around(e)), extent=_x(e), kappa=kappa_of(n), csw=0.0, precision=fmt(n > 20_000),
                    ncol=rng.choice([1, 3, 8, 12, 13, 16, 24]))
    if op in ("batch", "serve"):
        lat = [32, 16, 16, 16]
        parts = []
        for lo, hi, most in ((64, 1000, 12), (1000, 8000, 12), (8000, 30_000, 4)):
            parts.append("%s*%d" % (_x([min(x, l) for x, l in zip(box(lo, hi, 16), lat)]), rng.randint(1, most)))
        return dict(op=op, lattice=_x(lat), boxes=" ".join(parts), kappa=round(rng.uniform(0.130, 0.140), 4),
                    precision=rng.choice(["fp32"] * 3 + ["fp16"]))
    if op == "series":
        s = rng.choice([4, 6, 8, 12, 16])
        t = rng.choice([12, 16, 24, 32])
        inner = sorted(rng.sample(range(2, t), rng.randint(1, 3)))
        return dict(op=op, lattice=_x([t, s, s, s]), slabs=" ".join(map(str, inner + [t])),
                    kappa=round(rng.uniform(0.128, 0.138), 4), csw=0.0, precision=rng.choice(["fp32", "fp32", "fp16"]))
    if op == "expanded":
        e = box(256, 150_000)
        return dict(op=op, lattice=_x(around(e)), extent=_x(e), kappa=0.140, p=rng.choice([1, 2, 5, 8]),
                    ncol=rng.choice([1, 4, 12]))
    if op == "modes":
        e = box(1000, 20_000)
        return dict(op=op, lattice=_x(around(e)), extent=_x(e), kappa=round(rng.uniform(0.128, 0.138), 4),
                    precision="fp32", m=log_int(4, 64), iters=1)
    if op == "gram":
        e = box(2000, 80_000, 24)
        return dict(op=op, lattice=_x(around(e)), extent=_x(e), m=log_int(8, 128))
    e = box(1000, 30_000, 24)
    return dict(op=op, lattice=_x(around(e)), extent=_x(e), m=log_int(4, 40), form=rng.randrange(3))


def _x(v):
    return "x".join(str(int(i)) for i in v)


def _ints(s):
    return tuple(int(i) for i in s.split("x"))


# ------------------------------------------------------------------------- inputs

def _su3(lead, g, dev):
    """Links 1 + i eps H with Gaussian Hermitian H, orthonormalized: [..., 3, 3] complex128."""
    n = math.prod(lead)
    u = torch.empty((n, 3, 3), dtype=torch.complex128, device=dev)
    step = 1 << 21
    for a in range(0, n, step):
        h = torch.randn((min(n, a + step) - a, 8), dtype=torch.float64, device=dev, generator=g) * (0.5 * EPS)
        d = h[:, 7] / math.sqrt(3.0)
        r0 = torch.stack([torch.complex(torch.ones_like(d), h[:, 2] + d), torch.complex(h[:, 1], h[:, 0]),
                          torch.complex(h[:, 4], h[:, 3])], 1)
        r1 = torch.stack([torch.complex(-h[:, 1], h[:, 0]), torch.complex(torch.ones_like(d), d - h[:, 2]),
                          torch.complex(h[:, 6], h[:, 5])], 1)
        r0 = r0 / torch.linalg.vector_norm(r0, dim=1, keepdim=True)
        r1 = r1 - (r0.conj() * r1).sum(1, keepdim=True) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=1, keepdim=True)
        u[a:a + step] = torch.stack([r0, r1, torch.linalg.cross(r0, r1).conj()], 1)
    return u.reshape(tuple(lead) + (3, 3))


def _gauss(shape, g, dev):
    return torch.complex(torch.randn(shape, dtype=torch.float64, device=dev, generator=g),
                         torch.randn(shape, dtype=torch.float64, device=dev, generator=g))


def _noise(ncol, n, g, dev):
    """Spin-colour diluted noise columns (the first 12), Gaussian volume sources beyond."""
    eta = torch.zeros((ncol, n, 4, 3), dtype=torch.complex128, device=dev)
    z = _gauss((n,), g, dev) / math.sqrt(2.0)
    for c in range(min(ncol, 12)):
        eta[c, :, c // 3, c % 3] = z
    if ncol > 12:
        eta[12:] = _gauss((ncol - 12, n, 4, 3), g, dev)
    return eta


def _boxes(case):
    """(origin, extent) of every box of a batch, spread over the lattice."""
    lat, out = _ints(case["lattice"]), []
    for part in case["boxes"].split():
        ext, count = part.split("*")
        ext = _ints(ext)
        for k in range(int(count)):
            per = [max(1, l // x) for l, x in zip(lat, ext)]
            o, r = [], k
            for m in (3, 2, 1, 0):
                o.insert(0, (r % per[m]) * ext[m] if ext[m] < lat[m] else 0)
                r //= per[m]
            o[0] = (o[0] + r) % lat[0]
            out.append((tuple(o), ext))
    return out


def _slabs(case):
    lat = _ints(case["lattice"])
    return [(((0 if t == lat[0] else -(t // 2) % lat[0]), 0, 0, 0), (t,) + lat[1:])
            for t in map(int, case["slabs"].split())]


def _centre(o, e, lat):
    return tuple((a + b // 2) % l for a, b, l in zip(o, e, lat))


def _inputs(case, seed, dev):
    """Every input of a case from its seed (shared by prepare and exact)."""
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) * 7919 + 13)
    lat = _ints(case["lattice"])
    s = {"lat": lat}
    if case["op"] not in ("gram", "colourless"):
        s["U"] = _su3((4, math.prod(lat)), g, dev)
    if "extent" in case:
        s["o"] = _ints(case.get("origin", "0x0x0x0"))
        s["e"] = _ints(case["extent"])
        s["n"] = math.prod(s["e"])
    if case["op"] in ("noise", "expanded"):
        s["eta"] = _noise(case["ncol"], s["n"], g, dev)
    if case["op"] == "modes":
        s["V0"] = _gauss((case["m"], s["n"], 4, 3), g, dev)
    if case["op"] in ("gram", "colourless"):
        # solutions of the operator decay away from the cut: one amplitude per time slice
        amp = torch.exp(-0.5 * torch.arange(s["e"][0], dtype=torch.float64, device=dev)).repeat_interleave(
            s["n"] // s["e"][0])
        s["A"] = _gauss((case["m"], s["n"], 4, 3), g, dev) * amp.view(1, -1, 1, 1)
    return s


class State:
    """A context with its resident gauge field, the inputs and the output buffers."""

    def __init__(self, case, seed):
        self.ctx = ddp.ddp_create(0, torch.cuda.current_stream().cuda_stream)
        self.case = case
        i = _inputs(case, seed, "cuda")
        self.lat = lat = i["lat"]
        op = case["op"]
        # modes of a projector cut need a field only for the lattice they live on
        U = i["U"] if "U" in i else torch.eye(3, dtype=torch.complex128, device="cuda").expand(
            4, math.prod(lat), 3, 3).contiguous()
        self.gauge = ddp.ddp_load_gauge(self.ctx, U, lat, ddp.DDP_BC_ANTIPERIODIC)
        if op in ("batch", "serve"):
            self.boxes = _boxes(case)
        elif op == "series":
            self.boxes = _slabs(case)
        else:
            self.boxes = [(i["o"], i["e"])]
        self.dom = [ddp.ddp_set_domain(self.ctx, self.gauge, o, e) for o, e in self.boxes]
        self.src = [_centre(o, e, lat) for o, e in self.boxes]
        self.prec = PREC.get(case.get("precision"))

        def field(ncol, n):
            return torch.zeros((ncol, n, 4, 3), dtype=torch.complex128, device="cuda")

        sizes = [math.prod(e) for _, e in self.boxes]
        if op in ("propagator", "batch", "serve", "series"):
            self.S = [field(12, n) for n in sizes]
        if op == "serve":
            self.C = torch.zeros((len(self.boxes), 2 * lat[0]), dtype=torch.float64, device="cuda")
            ddp.ddp_serve_config(self.ctx, 4 << 30, 32, self.prec)
        if op == "series":
            self.src = (0, 0, 0, 0)
            self.C = torch.zeros((len(sizes), 4, 2 * lat[0]), dtype=torch.float64, device="cuda")
        if op in ("noise", "expanded"):
            self.eta = i["eta"]
            self.psi = torch.zeros_like(self.eta)
        if op == "expanded":
            self.C = torch.zeros(2 * lat[0], dtype=torch.float64, device="cuda")
        if op == "modes":
            self.V0 = i["V0"]
            self.V = torch.zeros_like(self.V0)
        if op in ("gram", "colourless"):
            self.A = i["A"]
            m = case["m"]
            shape = (lat[0], m, m) if op == "gram" else (lat[0], m, m, m, 4)
            self.M = torch.zeros(shape, dtype=torch.complex128, device="cuda")

    def __del__(self):
        if getattr(self, "ctx", None):
            ddp.ddp_destroy(self.ctx)
            self.ctx = None


def prepare(case, seed):
    return State(case, seed)


# ------------------------------------------------------------------------- one pass

def run(s):
    c, ctx, op = s.case, s.ctx, s.case["op"]
    if op == "propagator":
        ddp.ddp_solve_propagator(ctx, s.dom[0], c["kappa"], c["csw"], s.src[0], TOL, s.prec, s.S[0])
        return {"S": s.S[0]}
    if op == "noise":
        ddp.ddp_solve_sources(ctx, s.dom[0], c["kappa"], c["csw"], s.eta, c["ncol"], TOL, s.prec, s.psi)
        return {"psi": s.psi}
    if op == "batch":
        reqs = [ddp.make_req(d, c["kappa"], x, TOL, out) for d, x, out in zip(s.dom, s.src, s.S)]
        ddp.ddp_solve_batch(ctx, reqs, s.prec)
        return {"S": s.S}
    if op == "serve":
        todo = list(range(len(s.dom)))
        flying = {}
        while todo or flying:
            while todo:
                k = todo[0]
                rc, t = ddp.ddp_submit(ctx, ddp.make_req(s.dom[k], c["kappa"], s.src[k], TOL, s.S[k]))
                if rc != ddp.DDP_OK:
                    break
                flying[t] = todo.pop(0)
            ddp.ddp_serve_step(ctx)
            for t in list(flying):
                done, _ = ddp.ddp_poll(ctx, t)
                if done:
                    k = flying.pop(t)
                    ddp.ddp_contract(ctx, ddp.DDP_CONTRACT_NUCLEON, s.dom[k], s.S[k], s.C[k])
        return {"S": s.S, "C": s.C}
    if op == "series":
        mask = (1 << ddp.DDP_CONTRACT_PSEUDO_LOCAL) | (1 << ddp.DDP_CONTRACT_NUCLEON) | (1 << ddp.DDP_CONTRACT_PION)
        ddp.ddp_propagator_series(ctx, s.dom, c["kappa"], s.src, TOL, s.prec, S_out=s.S,
                                  contract_mask=mask, C_out=s.C, csw=c["csw"])
        return {"S": s.S, "C": s.C}
    if op == "expanded":
        ddp.ddp_hop_power(ctx, s.dom[0], c["kappa"], c["p"], s.eta, s.psi, c["ncol"])
        ddp.ddp_contract(ctx, ddp.DDP_CONTRACT_PSEUDO_NOISE, s.dom[0], s.psi, s.C, eta=s.eta, ncol=c["ncol"])
        return {"psi": s.psi, "C": s.C}
    if op == "modes":
        s.V.copy_(s.V0)
        ddp.ddp_inverse_iteration(ctx, s.dom[0], c["kappa"], s.V, c["m"], c["iters"], TOL, s.prec)
        return {"V": s.V}
    if op == "gram":
        ddp.ddp_gram_slices(ctx, s.dom[0], s.A, c["m"], s.M)
        return {"M": s.M}
    ddp.ddp_colourless_slices(ctx, s.dom[0], s.A, c["m"], c["form"], s.M)
    return {"X": s.M}


# ------------------------------------------------------------------------- what a pass needs

def work(case):
    """Links of the domain and sources read once, results written once; for solves the
    operations of one application of D per column (1320 per site and column and a few more:
    the residual that every solve has to check), the iterations not counted."""
    op = case["op"]
    if op in ("batch", "serve"):
        sizes = [math.prod(e) for _, e in _boxes(case)]
    elif op == "series":
        sizes = [math.prod(e) for _, e in _slabs(case)]
    else:
        sizes = [math.prod(_ints(case["extent"]))]
    n = sum(sizes)
    links, spinor, dirac = 4 * 144, 192, 1368
    if op in ("propagator", "batch", "serve", "series"):
        return {"bytes": n * (links + 12 * spinor), "flops": n * 12 * dirac}
    if op == "series":
        return {"bytes": n * (links + 12 * spinor) , "flops": n * 12 * dirac}
    if op == "noise":
        return {"bytes": n * (links + 2 * case["ncol"] * spinor), "flops": n * case["ncol"] * dirac}
    if op == "expanded":
        return {"bytes": n * (links + 2 * case["ncol"] * spinor), "flops": n * case["ncol"] * dirac * case["p"]}
    m = case["m"]
    if op == "modes":
        return {"bytes": n * (links + 2 * m * spinor), "flops": n * m * (dirac + 4 * 12 * 8 * m)}
    lat = _ints(case["lattice"])
    if op == "gram":
        return {"bytes": n * m * spinor + lat[0] * m * m * 16, "flops": n * 12 * m * m * 4}
    return {"bytes": n * m * spinor + lat[0] * m ** 3 * 64, "flops": n * m * (m + 1) // 2 * m * 4 * 3 * 8}


# ------------------------------------------------------------------------- 64-bit values

class _Exact:
    """The Dirac operator of a box and the contractions, in plain torch at 64 bits."""

    def __init__(self, U, lat, kappa, csw=0.0):
        self.U, self.lat, self.kappa, self.csw, self.dev = U, lat, kappa, csw, U.device
        z, i2 = torch.zeros((2, 2), dtype=torch.complex128), torch.eye(2, dtype=torch.complex128)
        sig = [torch.tensor(v, dtype=torch.complex128) for v in
               ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]])]

        def blocks(a, b):
            return torch.cat([torch.cat([z, a], 1), torch.cat([b, z], 1)], 0).to(self.dev)

        self.gamma = [blocks(i2, i2)] + [blocks(-1j * t, 1j * t) for t in sig]
        self.clover = self._clover() if csw else None

    def _clover(self):
        """c_sw (i/4) sum sigma_{mu nu} F_{mu nu}(x), [V, 3, 4, 3, 4] over (colour, spin)."""
        lat = self.lat
        u = self.U.reshape((4,) + lat + (3, 3))

        def at(mu, x):
            t = u[mu]
            for m, d in x.items():
                if d:
                    t = torch.roll(t, -d, dims=m)
            return t

        def dag(t):
            return t.conj().transpose(-1, -2)

        out = torch.zeros((math.prod(lat), 3, 4, 3, 4), dtype=torch.complex128, device=self.dev)
        for a in range(4):
            for b in range(a + 1, 4):
                q = at(a, {}) @ at(b, {a: 1}) @ dag(at(a, {b: 1})) @ dag(at(b, {}))
                q = q + at(b, {}) @ dag(at(a, {a: -1, b: 1})) @ dag(at(b, {a: -1})) @ at(a, {a: -1})
                q = q + dag(at(a, {a: -1})) @ dag(at(b, {a: -1, b: -1})) @ at(a, {a: -1, b: -1}) @ at(b, {b: -1})
                q = q + dag(at(b, {b: -1})) @ at(a, {b: -1}) @ at(b, {a: 1, b: -1}) @ dag(at(a, {}))
                f = ((q - dag(q)) / 8).reshape(-1, 3, 3)
                s = 0.5j * (self.gamma[a] @ self.gamma[b] - self.gamma[b] @ self.gamma[a])
                out += 0.5j * self.csw * torch.einsum("xab,st->xasbt", f, s)
        return out

    def domain(self, o, e):
        """Neighbour tables of a box: per hop (neighbour, factor, oriented links)."""
        lat, dev = self.lat, self.dev
        k = torch.stack(torch.meshgrid(*[torch.arange(x, device=dev) for x in e], indexing="ij"), -1).reshape(-1, 4)
        L, O, E = (torch.tensor(v, device=dev) for v in (lat, o, e))

        def lex(c, dims):
            return ((c[:, 0] * dims[1] + c[:, 1]) * dims[2] + c[:, 2]) * dims[3] + c[:, 3]

        x = (O + k) % L
        self.rows = lex(x, lat)
        self.slice = x[:, 0]
        self.hops = []
        for mu in range(4):
            for d in (1, -1):
                kn = k.clone()
                kn[:, mu] += d
                ok = torch.ones(len(k), dtype=torch.bool, device=dev)
                if e[mu] < lat[mu]:
                    ok = (kn[:, mu] >= 0) & (kn[:, mu] < e[mu])
                kn = kn % E
                f = ok.to(torch.float64)
                if mu == 0:
                    f = torch.where(x[:, 0] == (lat[0] - 1 if d == 1 else 0), -f, f)
                xb = x.clone()
                if d == -1:
                    xb[:, mu] = (xb[:, mu] - 1) % lat[mu]
                u = self.U[mu][lex(xb, lat)]
                if d == -1:
                    u = u.conj().transpose(-1, -2)
                u = u * f.view(-1, 1, 1)
                spin = torch.eye(4, dtype=torch.complex128, device=dev) - d * self.gamma[mu]
                self.hops.append((lex(kn, e), u.contiguous(), spin))

    def hop(self, v):
        """D_hop v on [site, colour, spin, column]."""
        n, _, _, c = v.shape
        out = torch.zeros_like(v)
        for nb, u, spin in self.hops:
            w = (u @ v[nb].reshape(n, 3, 4 * c)).reshape(n * 3, 4, c)
            out += (spin @ w).reshape(n, 3, 4, c)
        return out

    def dirac(self, v):
        out = v / (2 * self.kappa) - 0.5 * self.hop(v)
        if self.clover is not None:
            n, _, _, c = v.shape
            out += (self.clover[self.rows].reshape(n, 12, 12) @ v.reshape(n, 12, c)).reshape(v.shape)
        return out

    def solve(self, b):
        """BiCGStab on all columns, restarted on the true residual until it stops falling."""
        x = torch.zeros_like(b)
        bn = torch.linalg.vector_norm(b, dim=(0, 1, 2))

        def dot(p, q):
            return (p.conj() * q).sum((0, 1, 2))

        def ratio(p, q, live):
            """p / q of the live columns, 0 elsewhere and where the recurrence breaks down."""
            out = p / torch.where(live & (q.abs() > 0), q, torch.ones_like(q))
            return torch.where(live & (q.abs() > 0) & torch.isfinite(out.abs()), out, torch.zeros_like(out))

        for _ in range(6):
            r = b - self.dirac(x)
            rn0 = torch.linalg.vector_norm(r, dim=(0, 1, 2))
            live = rn0 > 1e-15 * bn
            if not bool(live.any()):
                break
            rh, p, rho, dx = r.clone(), r.clone(), dot(r, r), torch.zeros_like(x)
            for it in range(2000):
                v = self.dirac(p)
                alpha = ratio(rho, dot(rh, v), live)
                r = r - alpha * v
                t = self.dirac(r)
                omega = ratio(dot(t, r), dot(t, t), live)
                dx = dx + alpha * p + omega * r
                r = r - omega * t
                # a column stops when it has converged or its recurrence has broken down
                live = live & (torch.linalg.vector_norm(r, dim=(0, 1, 2)) > 1e-7 * rn0) & (omega.abs() > 0)
                if it % 8 == 7 and not bool(live.any()):
                    break
                new = dot(rh, r)
                beta = ratio(new, rho, live) * ratio(alpha, omega, live)
                p = r + beta * (p - omega * v)
                rho = new
            x = x + dx
            worst = float((torch.linalg.vector_norm(b - self.dirac(x), dim=(0, 1, 2)) / bn).max())
            if worst < 1e-14:
                break
        return x

    @staticmethod
    def inside(v):      # [column, site, spin, colour] -> [site, colour, spin, column]
        return v.permute(1, 3, 2, 0).contiguous()

    @staticmethod
    def outside(v):
        return v.permute(3, 0, 2, 1).contiguous()

    def propagator(self, o, e, src):
        self.domain(o, e)
        k = [(a - b) % l for a, b, l in zip(src, o, self.lat)]
        at = ((k[0] * e[1] + k[1]) * e[2] + k[2]) * e[3] + k[3]
        b = torch.zeros((math.prod(e), 3, 4, 12), dtype=torch.complex128, device=self.dev)
        for c in range(12):
            b[at, c % 3, c // 3, c] = 1
        return self.outside(self.solve(b)), at

    def by_slice(self, w):
        """Sum of a site field over every global time slice, as interleaved reals."""
        out = torch.zeros(self.lat[0], dtype=torch.complex128, device=self.dev)
        out.index_add_(0, self.slice, w)
        return torch.view_as_real(out).reshape(-1)

    def noise_trace(self, eta, psi):
        g5 = torch.tensor([-1.0, -1.0, 1.0, 1.0], dtype=torch.float64, device=self.dev).view(1, 1, 4, 1)
        return self.by_slice((eta.conj() * g5 * psi).sum((0, 2, 3)))

    def nucleon(self, S):
        n = S.shape[1]
        s = S.reshape(4, 3, n, 4, 3)          # [source spin b, source colour b, site, spin, colour]
        G = torch.zeros((4, 4), dtype=torch.complex128, device=self.dev)
        G[0, 1], G[1, 0], G[2, 3], G[3, 2] = -1j, 1j, -1j, 1j
        P = 0.5 * (torch.eye(4, dtype=torch.complex128, device=self.dev) - self.gamma[0])

        def m(a, b):                          # spin matrix [site, sink, source] of colours (a, b)
            return s[:, b, :, :, a].permute(1, 2, 0)

        perms = [((0, 1, 2), 1), ((1, 2, 0), 1), ((2, 0, 1), 1), ((0, 2, 1), -1), ((2, 1, 0), -1), ((1, 0, 2), -1)]
        w = torch.zeros(n, dtype=torch.complex128, device=self.dev)
        for (a, b, c), s1 in perms:
            for (f, e, g), s2 in perms:
                first = (m(a, g) * (G @ m(b, f) @ G)).sum((1, 2)) * (m(c, e) * P.T).sum((1, 2))
                second = (m(a, g) * (G @ m(b, e) @ P @ m(c, f) @ G)).sum((1, 2))
                w += s1 * s2 * (first - second)
        return self.by_slice(w)


def _qr(V):
    """The orthonormal columns Gram-Schmidt gives: V [m, ...] complex."""
    q, r = torch.linalg.qr(V.reshape(V.shape[0], -1).T)
    d = torch.diagonal(r)
    return (q * (d / d.abs())).T.reshape(V.shape).contiguous()


def exact(case, seed):
    op = case["op"]
    if op in ("batch", "serve"):
        sc = 12 * sum(math.prod(e) for _, e in _boxes(case))
    elif op == "series":
        sc = 12 * sum(math.prod(e) for _, e in _slabs(case))
    else:
        sc = math.prod(_ints(case["extent"])) * case.get("ncol", case.get("m", 12))
    if op in ("propagator", "noise", "batch", "serve", "series", "modes") and sc > EXACT_SITE_COLS:
        return None
    if op in ("batch", "serve") and len(_boxes(case)) > 24:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    i = _inputs(case, seed, dev)
    lat = i["lat"]
    if op == "gram":
        A = i["A"].reshape(case["m"], i["e"][0], -1)
        M = torch.zeros((lat[0], case["m"], case["m"]), dtype=torch.complex128, device=dev)
        for t in range(i["e"][0]):
            M[(i["o"][0] + t) % lat[0]] = A[:, t].conj() @ A[:, t].T
        return {"M": M}
    if op == "colourless":
        m = case["m"]
        A = i["A"].reshape(m, i["e"][0], -1, 4, 3)
        if case["form"] == 1:
            A = A.conj() * torch.tensor([-1.0, -1.0, 1.0, 1.0], dtype=torch.float64, device=dev).view(1, 1, 1, 4, 1)
        elif case["form"] == 2:
            A = -A
        X = torch.zeros((lat[0], m, m, m, 4), dtype=torch.complex128, device=dev)
        for t in range(i["e"][0]):
            a = A[:, t]
            s = (a.permute(3, 1, 0, 2).reshape(3, -1, 4 * m))                    # [colour][site][(k, alpha)]
            for j in range(m):
                acc = 0
                for c in range(3):
                    p, q = (c + 1) % 3, (c + 2) % 3

                    def f(u, v):                                                # (s_i^u)^T C g5 s_j^v, all i
                        b = a[j, :, :, v]
                        return 1j * (a[:, :, 1, u] * b[:, 0] - a[:, :, 0, u] * b[:, 1]
                                     + a[:, :, 3, u] * b[:, 2] - a[:, :, 2, u] * b[:, 3])
                    acc = acc + (f(p, q) - f(q, p)) @ s[c]
                X[(i["o"][0] + t) % lat[0], :, j] = acc.reshape(m, m, 4)
        return {"X": X}
    x = _Exact(i["U"], lat, case["kappa"], case.get("csw", 0.0))
    if op == "propagator":
        return {"S": x.propagator(i["o"], i["e"], _centre(i["o"], i["e"], lat))[0]}
    if op == "noise":
        x.domain(i["o"], i["e"])
        return {"psi": x.outside(x.solve(x.inside(i["eta"])))}
    if op == "expanded":
        x.domain(i["o"], i["e"])
        v = x.inside(i["eta"])
        for _ in range(case["p"]):
            v = case["kappa"] * x.hop(v)
        v = x.outside(v)
        return {"psi": v, "C": x.noise_trace(i["eta"], v)}
    if op == "modes":
        x.domain(i["o"], i["e"])
        V = _qr(i["V0"])
        for _ in range(case["iters"]):
            V = _qr(x.outside(x.solve(x.inside(V))))
        return {"V": V}
    if op in ("batch", "serve"):
        S, C = [], []
        for o, e in _boxes(case):
            S.append(x.propagator(o, e, _centre(o, e, lat))[0])
            C.append(x.nucleon(S[-1]))
        return {"S": S} if op == "batch" else {"S": S, "C": torch.stack(C)}
    # nested domains of one source: propagators and correlators
    S = []
    C = torch.zeros((len(_slabs(case)), 4, 2 * lat[0]), dtype=torch.float64, device=dev)
    for q, (o, e) in enumerate(_slabs(case)):
        s, at = x.propagator(o, e, (0, 0, 0, 0))
        S.append(s)
        diag = torch.einsum("sasa->s", s[:, at].reshape(4, 3, 4, 3))
        C[q, ddp.DDP_CONTRACT_PSEUDO_LOCAL, :2] = torch.view_as_real(diag[2] + diag[3] - diag[0] - diag[1])
        C[q, ddp.DDP_CONTRACT_NUCLEON] = x.nucleon(s)
        C[q, ddp.DDP_CONTRACT_PION] = x.by_slice((s.conj() * s).sum((0, 2, 3)))
    return {"S": S, "C": C}
