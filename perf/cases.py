"""Performance cases: the calls that a user of the framework makes, over the sizes they are made at.

A case names one kind of call and its sizes.  `prepare` makes the inputs on the GPU from the seed (a two-disk galaxy,
closed-form potentials) and the context a program keeps; `run` is one pass through the public entry points; `exact`
is the same result in 64 bits from plain torch, without the package: the discrete Poisson problems by sine
transforms, everything else by its definition."""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as nnf

G, A0 = 4.30e-3, 3.6
SHIFT = 24  # fixed-point scale of the deposit, 2^24 units per solar mass
F64 = torch.float64


def listed():
    return [
        # a quick look at a model: the smallest grid, the library's default precision; latency is all there is
        dict(name="newton-33", kind="solve", eq="newton", n=32, box=0, sets=1, precision="mixed", rel_tol=1e-10, dc=2,
             ncycle=1, particles=20000),
        # the rotation curve of a solved galaxy: a post-processing call of one small launch
        dict(name="curve-129x2", kind="curve", n=128, nboxes=2, nbins=50, nphi=64),
        # an inner box at the paper's middle grid, default precision (FP64 defect correction)
        dict(name="newton-129-mixed", kind="solve", eq="newton", n=128, box=1, sets=1, precision="mixed", rel_tol=1e-10,
             dc=2, ncycle=1, particles=200000),
        # the QUMOND solve of an inner box of the 257^3 workload, fixed-point defect correction
        dict(name="mond-257-fixed", kind="solve", eq="mond", n=256, box=1, sets=1, precision="fixed", rel_tol=1e-10,
             dc=4, ncycle=1, particles=0),
        # the Newtonian solve of the outermost box of the large workload
        dict(name="newton-513-fixed", kind="solve", eq="newton", n=512, box=0, sets=1, precision="fixed", rel_tol=1e-10,
             dc=2, ncycle=1, particles=4000001),
        # the paper's own algorithm: FP64, six V-cycles per full-multigrid level, no tolerance
        dict(name="paper-129-fp64", kind="solve", eq="newton", n=128, box=1, sets=1, precision="fp64", rel_tol=0.0, dc=2,
             ncycle=6, particles=200000),
        # a chunk of the rotation-curve fit sweep: eight parameter sets in each launch
        dict(name="mond-129x8-fixed", kind="solve", eq="mond", n=128, box=1, sets=8, precision="fixed", rel_tol=1e-8,
             dc=3, ncycle=1, particles=0),
        # the deposit of the two-disk workload's particles (a ragged count)
        dict(name="deposit-257", kind="deposit", n=256, box=1, particles=1999993),
        # the QUMOND source of a 257^3 box
        dict(name="source-257", kind="source", n=256, box=1),
        # the forces at every particle of the two-disk workload
        dict(name="forces-257x3", kind="forces", n=256, nboxes=3, points=1999993),
        # the whole path as the headline benchmark runs it: deposits, far field, six solves, sources, forces, curve
        dict(name="two-disk-257x3", kind="whole", n=256, nboxes=3, particles=2000000, nbins=50, nphi=64, dc=4),
        # a training step of the learned initial guess: forward and backward of a batch
        dict(name="guess-gradients-64", kind="guess", S=64, batch=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(("solve", "deposit", "source", "forces", "curve", "whole", "guess"), (8, 2, 1, 2, 1, 2, 1))[0]
    if kind == "solve":
        precision = rng.choices(("fixed", "mixed", "fp64"), (3, 2, 1))[0]
        n = rng.choice((32, 64, 128, 256) if precision != "fp64" else (32, 64, 128))
        sets = rng.randint(1, {32: 24, 64: 16, 128: 10, 256: 2}[n]) if rng.random() < 0.5 else 1
        eq = rng.choice(("newton", "mond"))
        paper = rng.random() < 0.2
        return dict(kind=kind, eq=eq, n=n, box=rng.randint(0, 2), sets=sets, precision=precision,
                    rel_tol=0.0 if paper else float("%.1e" % 10.0 ** rng.uniform(-10.0, -7.0)), dc=rng.randint(1, 4),
                    ncycle=rng.choice((2, 6)) if paper else 1,
                    particles=_log_int(rng, 2e4, 1e6) if eq == "newton" else 0)
    if kind == "deposit":
        return dict(kind=kind, n=rng.choice((64, 128, 256)), box=rng.randint(0, 2), particles=_log_int(rng, 1e4, 1e7))
    if kind == "source":
        return dict(kind=kind, n=rng.choice((32, 64, 128, 256)), box=rng.randint(0, 5))
    if kind == "forces":
        return dict(kind=kind, n=rng.choice((64, 128, 256)), nboxes=rng.randint(1, 4), points=_log_int(rng, 1e3, 5e6))
    if kind == "curve":
        return dict(kind=kind, n=rng.choice((64, 128)), nboxes=rng.randint(1, 4), nbins=rng.randint(10, 200),
                    nphi=rng.randint(16, 256))
    if kind == "whole":
        return dict(kind=kind, n=rng.choice((64, 128)), nboxes=rng.randint(2, 3), particles=_log_int(rng, 1e5, 2e6),
                    nbins=rng.randint(20, 60), nphi=64, dc=rng.randint(2, 4))
    return dict(kind=kind, S=rng.choice((16, 32, 48, 64)), batch=rng.randint(1, 3))


# --- inputs ---------------------------------------------------------------------------------------------------------
def _side0(case):
    """Side of box 0 (pc): 120 kpc as the 257^3 workload, 240 kpc on the 513^3 grid, 80 kpc below."""
    n = case.get("n", 64)
    return 240000.0 if n > 256 else (120000.0 if n == 256 else 80000.0)


def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + salt * 7919 + 17) & 0x7FFFFFFF)


def _galaxy(count, seed, salt=0):
    """Stellar and gas exponential disks (sech^2 heights), half of the particles each, in random order of radius."""
    g = _gen(seed, salt)
    u = torch.rand(5, count, dtype=F64, device="cuda", generator=g).clamp_(1e-12, 1.0 - 1e-12)
    star = torch.arange(count, device="cuda") < (count + 1) // 2
    hs = 300.0 + 300.0 * float(torch.rand(1, dtype=F64, device="cuda", generator=g))
    R = -torch.log(u[0] * u[1]) * torch.where(star, 3000.0, 8000.0)
    z = torch.atanh(2.0 * u[3] - 1.0) * torch.where(star, hs, 100.0)
    ph = 2.0 * math.pi * u[2]
    m_star = 2.0 * math.pi * 500.0 * 3000.0 ** 2 / max(1, (count + 1) // 2)
    m_gas = 1.0e9 / max(1, count // 2)
    m = torch.where(star, m_star, m_gas).to(F64)
    return R * torch.cos(ph), R * torch.sin(ph), z, m


def _disk_params(seed, salt):
    """Masses and scale lengths of a stellar and a gas disk (Miyamoto-Nagai), drawn around the workloads' galaxy."""
    u = torch.rand(4, dtype=F64, device="cuda", generator=_gen(seed, 100 + salt)).tolist()
    return ((2.8e10 * (0.6 + 0.8 * u[0]), 3000.0 * (0.8 + 0.4 * u[1]), 300.0 + 300.0 * u[2]),
            (1.0e9, 8000.0 * (0.8 + 0.4 * u[3]), 150.0))


def _disk_phi(prm, x, y, z):
    phi = 0.0
    for M, a, b in prm:
        phi = phi - G * M / torch.sqrt(x * x + y * y + (a + torch.sqrt(z * z + b * b)) ** 2)
    return phi


def _axis(n, L):
    return (torch.arange(n + 1, dtype=F64, device="cuda") * (L / n) - 0.5 * L)


def _disk_grid(prm, n, L):
    """The disks' potential on the nodes of a box, [k][j][i]."""
    a = _axis(n, L)
    return _disk_phi(prm, a[None, None, :], a[None, :, None], a[:, None, None])


def _cells(t, n):
    """Cell index and offset of index coordinates, and which lie in the box."""
    ok = torch.ones(t[0].shape, dtype=torch.bool, device="cuda")
    idx, off = [], []
    for v in t:
        ok &= (v >= 0) & (v < n)
        f = torch.floor(v)
        idx.append(f.clamp(0, n - 1).to(torch.int64))
        off.append(v - f)
    return idx, off, ok


def _deposit(parts, n, L):
    """Fixed-point cloud-in-cell grid (int64) and the density."""
    x, y, z, m = parts
    inv_h = n / L
    (i, j, k), (dx, dy, dz), ok = _cells([(v - (-0.5 * L)) * inv_h for v in (x, y, z)], n)
    i, j, k, dx, dy, dz, ms = (v[ok] for v in (i, j, k, dx, dy, dz, m * 2.0 ** SHIFT))
    q = torch.zeros((n + 1) ** 3, dtype=torch.int64, device="cuda")
    for c in (0, 1):
        for b in (0, 1):
            for a in (0, 1):
                w = ((ms * (dx if a else 1.0 - dx)) * (dy if b else 1.0 - dy)) * (dz if c else 1.0 - dz)
                q.index_add_(0, (i + a) + (n + 1) * ((j + b) + (n + 1) * (k + c)), torch.round(w).to(torch.int64))
    return q, q.to(F64) * (2.0 ** -SHIFT * (inv_h * inv_h * inv_h))


def _source(p, L):
    """The QUMOND source of a potential on the nodes of a box, [k][j][i]: face fluxes in 64 bits."""
    n = p.shape[0] - 1
    ih = n / L
    src = torch.zeros_like(p)
    inner = (slice(1, -1),) * 3
    for ax in range(3):
        def sl(d, s):  # the interior along the other axes, `s` along this one and d shifted by one along an axis
            out = [slice(1, -1)] * 3
            out[ax] = s
            for o, q in d.items():
                out[o] = slice(1 + q, n + q) if o != ax else out[o]
            return p[tuple(out)]
        lo, hi = slice(0, n), slice(1, n + 1)
        dn = sl({}, hi) - sl({}, lo)
        g2 = (dn * ih) ** 2
        for o in range(3):
            if o != ax:
                t = (sl({o: 1}, lo) - sl({o: -1}, lo)) + (sl({o: 1}, hi) - sl({o: -1}, hi))
                g2 = g2 + (t * (0.25 * ih)) ** 2
                del t
        flux = torch.where(g2 > 0, 0.5 + 0.5 * torch.sqrt(1.0 + 4.0 * A0 / torch.sqrt(g2)), torch.zeros_like(g2)) * dn
        src[inner] += flux.narrow(ax, 1, n - 1) - flux.narrow(ax, 0, n - 1)
        del dn, g2, flux
    return src.mul_(ih * ih)


def _context(case, **over):
    import paper_1201_3185_gb300 as q
    prec = dict(mixed=q.QUMOND_PREC_MIXED, fixed=q.QUMOND_PREC_MIXED_FIXED, fp64=q.QUMOND_PREC_FP64)
    kw = dict(n=case["n"], nboxes=case.get("nboxes", case.get("box", 0) + 1), L0=_side0(case), G=G, a0=A0,
              precision=prec[case.get("precision", "fixed")], rel_tol=case.get("rel_tol", 1e-10), max_vcycles=60,
              ncycle=case.get("ncycle", 1), dc_vcycles=case.get("dc", 2), nsets=case.get("sets", 1))
    kw.update(over)
    return q.Context(q.default_params(**kw))


def _solve_inputs(case, seed):
    """Right-hand sides and parent potentials of every set, (n+1)^3 each."""
    n, L = case["n"], _side0(case) / 2 ** case["box"]
    rhs, par = [], []
    for s in range(case["sets"]):
        prm = _disk_params(seed, s)
        if case["eq"] == "newton":
            rhs.append(_deposit(_galaxy(case["particles"], seed, s), n, L)[1])
        else:
            rhs.append(_source(_disk_grid(prm, n, L), L).reshape(-1))
        if case["box"] > 0:
            par.append(_disk_grid(prm, n, 2.0 * L).reshape(-1))
    return torch.cat(rhs), (torch.cat(par) if par else None)


def _weights(seed):
    """He-normal convolution weights, small biases, a small head: the network before training."""
    g = _gen(seed, 3)
    p = []
    for ci, co in LAYERS:
        p.append(torch.randn(27 * ci * co, device="cuda", generator=g) * math.sqrt(2.0 / (27 * ci)))
        p.append(0.01 * torch.randn(co, device="cuda", generator=g))
    p.append(torch.randn(16, device="cuda", generator=g) * math.sqrt(1.0 / 16))
    p.append(torch.zeros(1, device="cuda"))
    return torch.cat(p).float()


def _sample(S, seed, salt):
    """Channels of one box as the training set holds them: scaled density, potential and target, BF16."""
    prm = _disk_params(seed, salt)
    L = 80000.0
    a = _axis(S, L)[:S]
    x, y, z = a[None, None, :], a[None, :, None], a[:, None, None]
    R, h = torch.sqrt(x * x + y * y), L / S
    rho = 500.0 / (2.0 * prm[0][2]) * torch.exp(-R / prm[0][1]) / torch.cosh(z / prm[0][2]).clamp(max=1e100) ** 2
    phi = _disk_phi(prm, x, y, z)
    target = -0.3 * torch.sqrt(phi.abs() / 1.0e5) + 0.0 * x
    return torch.stack([(4.0 * math.pi * G * h * h / 1.0e5) * rho, phi / 1.0e5, target]).reshape(-1).to(torch.bfloat16)


def prepare(case, seed):
    import paper_1201_3185_gb300 as q
    kind = case["kind"]
    st = dict(case=case)

    def empty(count, dtype=F64):
        return torch.zeros(count, dtype=dtype, device="cuda")

    if kind == "guess":
        S = case["S"]
        st["net"] = q.Guess(S, 1.0e5)
        st["net"].qumond_guess_set_params(_weights(seed))
        st["samples"] = [_sample(S, seed, b) for b in range(case["batch"])]
        st["flags"] = [float(b % 2) for b in range(case["batch"])]
        st["grads"], st["loss"] = empty(q.Guess.num_params(), torch.float32), empty(1, torch.float32)
        return st
    n = case["n"]
    nodes = (n + 1) ** 3
    if kind == "whole":
        over = dict(bc_mode=q.QUMOND_BC_MULTIPOLE)
        st["parts"] = _galaxy(case["particles"], seed)
        st["pipe"] = q.Pipeline(_context(case, **over), ctx_mond=_context(case, **over))
        st["g"] = tuple(torch.empty_like(st["parts"][0]) for _ in range(3))
        return st
    st["ctx"] = _context(case)
    if kind == "solve":
        st["rhs"], st["parent"] = _solve_inputs(case, seed)
        st["phi"] = empty(nodes * case["sets"])
    elif kind == "deposit":
        st["parts"] = _galaxy(case["particles"], seed)
        st["q"], st["rho"] = empty(nodes, torch.int64), empty(nodes)
    elif kind == "source":
        st["phiN"] = _disk_grid(_disk_params(seed, 0), n, _side0(case) / 2 ** case["box"]).reshape(-1)
        st["src"] = empty(nodes)
    else:
        prm = _disk_params(seed, 0)
        st["phis"] = [_disk_grid(prm, n, _side0(case) / 2 ** b).reshape(-1) for b in range(case["nboxes"])]
        if kind == "forces":
            st["q"] = _galaxy(case["points"], seed)[:3]
            st["g"] = tuple(empty(case["points"]) for _ in range(3))
        else:
            st["r"], st["vc"] = empty(case["nbins"]), empty(case["nbins"])
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "guess":
        st["net"].qumond_guess_gradients(st["samples"], st["flags"], st["grads"], st["loss"])
        return dict(grads=st["grads"], loss=st["loss"])
    if kind == "whole":
        res = st["pipe"].run(*st["parts"], nbins=case["nbins"], rmax=_rmax(case), nphi=case["nphi"], forces=st["g"])
        return dict(phiN=list(st["pipe"].phiN), phi=list(st["pipe"].phi), g=list(st["g"]), r=res.r, vc=res.vc)
    ctx = st["ctx"]
    if kind == "solve":
        fn = ctx.qumond_solve_newton if case["eq"] == "newton" else ctx.qumond_solve_mond
        fn(case["box"], st["rhs"], st["parent"], st["phi"])
        return dict(phi=st["phi"])
    if kind == "deposit":
        ctx.qumond_deposit(case["box"], *st["parts"], st["q"], st["rho"])
        return dict(q=st["q"], rho=st["rho"])
    if kind == "source":
        ctx.qumond_source(case["box"], st["phiN"], st["src"])
        return dict(src=st["src"])
    if kind == "forces":
        ctx.qumond_forces(st["phis"], *st["q"], *st["g"])
        return dict(g=list(st["g"]))
    ctx.qumond_rotation_curve(st["phis"], case["nbins"], _rmax(case), case["nphi"], st["r"], st["vc"])
    return dict(r=st["r"], vc=st["vc"])


def _rmax(case):
    return 0.25 * _side0(case)


def work(case):
    kind = case["kind"]
    if kind == "guess":
        vox, flops = case["S"] ** 3, 0.0
        for l, (ci, co) in enumerate(LAYERS):
            lev = (0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0)[l]
            flops += 2.0 * 27 * ci * co * vox / 8 ** lev
        return dict(bytes=case["batch"] * 6.0 * vox + 8.0 * sum(27 * a * b + b for a, b in LAYERS),
                    flops=3.0 * case["batch"] * flops)
    nodes = float((case["n"] + 1) ** 3)

    def solve(tol, ncycle):  # V(2,2) cycles of about 60 operations a node on all levels; a factor of ten each
        cycles = ncycle if tol == 0.0 else 1 + max(1, math.ceil(-math.log10(tol)) - 3)
        return dict(bytes=16.0 * nodes, flops=8.0 / 7.0 * 60.0 * cycles * nodes)

    if kind == "solve":
        w = solve(case["rel_tol"], case["ncycle"])
        return dict(bytes=case["sets"] * w["bytes"], flops=case["sets"] * w["flops"])
    if kind == "deposit":
        return dict(bytes=32.0 * case["particles"] + 16.0 * nodes, flops=40.0 * case["particles"])
    if kind == "source":
        return dict(bytes=16.0 * nodes, flops=70.0 * nodes)
    if kind == "forces":
        return dict(bytes=48.0 * case["points"] + 8.0 * min(nodes * case["nboxes"], 32.0 * case["points"]),
                    flops=90.0 * case["points"])
    if kind == "curve":
        return dict(bytes=16.0 * case["nbins"] + 256.0 * case["nbins"] * case["nphi"],
                    flops=150.0 * case["nbins"] * case["nphi"])
    w = solve(1e-10, 1)
    nb = case["nboxes"]
    return dict(bytes=56.0 * case["particles"] + 16.0 * nodes * nb,
                flops=nb * (2.0 * w["flops"] + 70.0 * nodes + 40.0 * case["particles"]) + 90.0 * case["particles"])


# --- the results in 64 bits ------------------------------------------------------------------------------------------
def _dst(a, ax):
    """Sine transform of the first kind along an axis of n - 1 interior values: sum_j a_j sin(pi j k / n)."""
    a = a.movedim(ax, -1)
    z = torch.zeros_like(a[..., :1])
    f = torch.fft.rfft(torch.cat([z, a, z, -a.flip(-1)], dim=-1), dim=-1)
    return (-0.5 * f.imag[..., 1:a.shape[-1] + 1]).movedim(-1, ax)


def _poisson(f, u, L):
    """The 7-point Dirichlet problem: u holds the boundary values, its interior is replaced."""
    n = u.shape[0] - 1
    b = f[1:-1, 1:-1, 1:-1] * (L / n) ** 2
    for ax in range(3):
        inner = [slice(1, -1)] * 3
        for at, src in ((0, 0), (n - 2, n)):
            inner[ax] = src
            b.select(ax, at).sub_(u[tuple(inner)])
    lam = 2.0 * torch.cos(math.pi * torch.arange(1, n, dtype=F64, device="cuda") / n) - 2.0
    for ax in range(3):
        b = _dst(b, ax)
    b = b / (lam[None, None, :] + lam[None, :, None] + lam[:, None, None])
    for ax in range(3):
        b = _dst(b, ax) * (2.0 / n)
    u[1:-1, 1:-1, 1:-1] = b
    return u


def _from_parent(par):
    """Values of the box of half the side at its own nodes, by trilinear interpolation of its parent."""
    n = par.shape[0] - 1
    v = par
    for ax in range(3):
        v = v.narrow(ax, n // 4, n // 2 + 1)
        up = torch.zeros([n + 1 if a == ax else v.shape[a] for a in range(3)], dtype=F64, device="cuda")
        even, odd = [slice(None)] * 3, [slice(None)] * 3
        even[ax], odd[ax] = slice(0, None, 2), slice(1, None, 2)
        up[tuple(even)] = v
        up[tuple(odd)] = 0.5 * (v.narrow(ax, 0, n // 2) + v.narrow(ax, 1, n // 2))
        v = up
    return v.contiguous()


def _grid(a, n):
    return a.reshape(n + 1, n + 1, n + 1)


def _forces(phis, n, L0, pts, first=None):
    """-grad phi at points: central differences at the nodes, cloud-in-cell weights, the finest box whose cell has
    interior corners only.  first: the finest box that a point may use."""
    out = [torch.zeros_like(pts[0]) for _ in range(3)]
    todo = torch.ones(pts[0].shape, dtype=torch.bool, device="cuda")
    for b in range(len(phis) - 1, -1, -1):
        L, p = L0 / 2 ** b, phis[b].reshape(-1)
        t = [(v + 0.5 * L) * (n / L) for v in pts]
        use = todo.clone() if first is None else todo & (first >= b)
        for v in t:
            use &= (v >= 1) & (v < n - 1)
        sel = use.nonzero().reshape(-1)
        (i, j, k), d, _ = _cells([v[sel] for v in t], n)
        g = [torch.zeros(sel.shape, dtype=F64, device="cuda") for _ in range(3)]
        for c in range(8):
            s = (c & 1, (c >> 1) & 1, c >> 2)
            o = (i + s[0]) + (n + 1) * ((j + s[1]) + (n + 1) * (k + s[2]))
            w = 1.0
            for a in range(3):
                w = w * (d[a] if s[a] else 1.0 - d[a])
            for a, step in enumerate((1, n + 1, (n + 1) ** 2)):
                g[a] += w * (p[o + step] - p[o - step]) * (-0.5 * n / L)
        for a in range(3):
            out[a][sel] = g[a]
        todo &= ~use
    return out


def _curve(phis, n, L0, nbins, rmax, nphi):
    R = (torch.arange(nbins, dtype=F64, device="cuda") + 0.5) * rmax / nbins
    t = 2.0 * math.pi * torch.arange(nphi, dtype=F64, device="cuda") / nphi
    c, s = torch.cos(t), torch.sin(t)
    x, y = (R[:, None] * c).reshape(-1), (R[:, None] * s).reshape(-1)
    first = torch.zeros(nbins, dtype=torch.int64, device="cuda")
    for b in range(len(phis)):
        first[R < 0.2 * L0 / 2 ** b] = b
    g = _forces(phis, n, L0, (x, y, torch.zeros_like(x)), first[:, None].expand(-1, nphi).reshape(-1))
    v2 = R * -(g[0].reshape(nbins, nphi) * c + g[1].reshape(nbins, nphi) * s).mean(dim=1)
    return R, torch.sign(v2) * torch.sqrt(v2.abs())


def _faces(n):
    m = torch.ones(n + 1, n + 1, n + 1, dtype=torch.bool, device="cuda")
    m[1:-1, 1:-1, 1:-1] = False
    return m


def _far_field(rho, n, L):
    """Boundary values of box 0: the exterior multipole series to degree 8 of the node masses about their centre, and
    the QUMOND potential of the total mass as a point there.  Two grids, zero inside."""
    deg = 8
    a = _axis(n, L)
    sel = (rho.reshape(-1) != 0).nonzero().reshape(-1)
    m = rho.reshape(-1)[sel] * (L / n) ** 3
    P = n + 1
    pos = [a[sel % P], a[(sel // P) % P], a[sel // (P * P)]]
    M = m.sum()
    com = [(m * v).sum() / M for v in pos]
    x, y, z = (v - c for v, c in zip(pos, com))
    xy, r2 = torch.complex(x, y), x * x + y * y + z * z

    def ladder(start, diag, step):  # terms (l, m), 0 <= m <= l <= deg, of a solid-harmonic recurrence
        top = start
        for mm in range(deg + 1):
            if mm:
                top = top * diag(mm)
            prev, cur = torch.zeros_like(top), top
            yield mm, mm, cur
            for l in range(mm, deg):
                prev, cur = cur, step(l, mm, cur, prev)
                yield l + 1, mm, cur

    mom = {}
    for l, mm, v in ladder(torch.ones_like(xy), lambda q: -xy / (2.0 * q),
                           lambda l, q, c, p: ((2 * l + 1) * z * c - r2 * p) / ((l + 1 - q) * (l + 1 + q))):
        mom[l, mm] = (m * v).sum()
    face = _faces(n)
    sel = face.reshape(-1).nonzero().reshape(-1)
    X, Y, Z = (v - c for v, c in zip((a[sel % P], a[(sel // P) % P], a[sel // (P * P)]), com))
    XY, R2 = torch.complex(X, Y), X * X + Y * Y + Z * Z
    R = torch.sqrt(R2)
    val = torch.zeros_like(X)
    for l, mm, v in ladder(torch.complex(1.0 / R, torch.zeros_like(R)), lambda q: -(2 * q - 1) * XY / R2,
                           lambda l, q, c, p: ((2 * l + 1) * Z * c - (l * l - q * q) * p) / R2):
        val += (1.0 if mm == 0 else 2.0) * (mom[l, mm].conj() * v).real
    A = G * M
    C = 4.0 * A0 * A
    mond = -A / (2.0 * R) + 0.5 * (-torch.sqrt(A * A + C * R2) / R + torch.sqrt(C) * torch.asinh(torch.sqrt(C) * R / A))
    out = [torch.zeros(P ** 3, dtype=F64, device="cuda") for _ in range(2)]
    out[0][sel], out[1][sel] = -G * val, mond
    return [_grid(o, n) for o in out]


def _exact_whole(case, seed):
    n, L0 = case["n"], _side0(case)
    parts = _galaxy(case["particles"], seed)
    phiN, phi = [], []
    for b in range(case["nboxes"]):
        L = L0 / 2 ** b
        rho = _grid(_deposit(parts, n, L)[1], n)
        bn, bm = _far_field(rho, n, L) if b == 0 else (_from_parent(phiN[-1]), _from_parent(phi[-1]))
        phiN.append(_poisson(4.0 * math.pi * G * rho, bn, L))
        phi.append(_poisson(_source(phiN[-1], L), bm, L))
    g = _forces(phi, n, L0, parts[:3])
    r, vc = _curve(phi, n, L0, case["nbins"], _rmax(case), case["nphi"])
    return dict(phiN=[p.reshape(-1) for p in phiN], phi=[p.reshape(-1) for p in phi], g=g, r=r, vc=vc)


# (cin, cout) of the network's 14 convolutions: encoder levels 0-3, decoder levels 2-0
LAYERS = ((16, 16), (16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128), (192, 64), (64, 64),
          (96, 32), (32, 32), (48, 16), (16, 16))


def _exact_guess(case, seed):
    """Loss and gradients of the network with its BF16 weights, everything else in 64 bits."""
    S = case["S"]
    p = _weights(seed).to(F64)
    leaves, o = [], 0
    for ci, co in LAYERS:
        w = p[o:o + 27 * ci * co].float().to(torch.bfloat16).to(F64).reshape(co, 27, ci).requires_grad_()
        o += 27 * ci * co
        leaves += [w, p[o:o + co].clone().requires_grad_()]
        o += co
    leaves += [p[o:o + 16].clone().requires_grad_(), p[o + 16:].clone().requires_grad_()]

    def conv(l, x):
        ci, co = LAYERS[l]
        w = leaves[2 * l].reshape(co, 3, 3, 3, ci).permute(0, 4, 1, 2, 3).contiguous()
        return torch.relu(nnf.conv3d(x, w, leaves[2 * l + 1], padding=1))

    def up(x):
        return nnf.interpolate(x, scale_factor=2, mode="nearest")

    total = 0.0
    for b in range(case["batch"]):
        ch = _sample(S, seed, b).to(F64).reshape(3, S, S, S)
        x = torch.zeros(1, 16, S, S, S, dtype=F64, device="cuda")
        x[0, 0], x[0, 1], x[0, 2] = ch[0], ch[1], float(b % 2)
        e0 = conv(1, conv(0, x))
        e1 = conv(3, conv(2, nnf.avg_pool3d(e0, 2)))
        e2 = conv(5, conv(4, nnf.avg_pool3d(e1, 2)))
        d = conv(7, conv(6, nnf.avg_pool3d(e2, 2)))
        d = conv(9, conv(8, torch.cat([up(d), e2], dim=1)))
        d = conv(11, conv(10, torch.cat([up(d), e1], dim=1)))
        d = conv(13, conv(12, torch.cat([up(d), e0], dim=1)))
        y = torch.einsum("c,czyx->zyx", leaves[-2], d[0]) + leaves[-1]
        total = total + ((y - ch[2]) ** 2).mean()
    total = total / case["batch"]
    total.backward()
    return dict(grads=torch.cat([t.grad.reshape(-1) for t in leaves]), loss=total.detach().reshape(1))


def exact(case, seed):
    kind = case["kind"]
    if kind == "guess":
        return _exact_guess(case, seed)
    if kind == "whole":
        return _exact_whole(case, seed)
    n, L0 = case["n"], _side0(case)
    L = L0 / 2 ** case.get("box", 0)
    if kind == "solve":
        rhs, par = _solve_inputs(case, seed)
        coef = 4.0 * math.pi * G if case["eq"] == "newton" else 1.0
        out = []
        for s in range(case["sets"]):
            cut = slice(s * (n + 1) ** 3, (s + 1) * (n + 1) ** 3)
            u = _from_parent(_grid(par[cut], n)) if par is not None else _grid(torch.zeros_like(rhs[cut]), n)
            out.append(_poisson(coef * _grid(rhs[cut], n), u, L).reshape(-1))
        return dict(phi=torch.cat(out))
    if kind == "deposit":
        q, rho = _deposit(_galaxy(case["particles"], seed), n, L)
        return dict(q=q, rho=rho)
    prm = _disk_params(seed, 0)
    if kind == "source":
        return dict(src=_source(_disk_grid(prm, n, L), L).reshape(-1))
    phis = [_disk_grid(prm, n, L0 / 2 ** b).reshape(-1) for b in range(case["nboxes"])]
    if kind == "forces":
        return dict(g=_forces(phis, n, L0, _galaxy(case["points"], seed)[:3]))
    r, vc = _curve(phis, n, L0, case["nbins"], _rmax(case), case["nphi"])
    return dict(r=r, vc=vc)
