"""The work that users of the library have it do, as cases that can be timed and compared.

A case is a dict of plain values: `kind` (what is called), the system (`geometry`, `natoms`,
`nchi`, and `grid` for the potential) and the options of the call. A program keeps one Context
per system and calls it with many response kernels, so the synthetic system and its context
belong to the case and are kept between preparations; the kernels, potentials, densities and
training rows come from the seed. Everything a call reads and writes is on the GPU, as in a
solver loop.

A TDDFT_MIXED context computes in single precision and returns its numbers in float64 arrays; a
program that asked for it keeps them as float32, and so does run().
"""
import dataclasses
import functools
import math

import numpy as np
import torch

from paper_1507_08157_gb300 import synthetic, tddft

DEV = "cuda"


def listed():
    return [
        # the smallest workload (8 atoms, 48^3) in the default precision, one state: launches, waits
        {"name": "apply_small8_fp64", "kind": "apply", "geometry": "small", "natoms": 8, "nchi": 4, "k": 1,
         "precision": "fp64"},
        # its solver with every default option: a random start and the first ten iterations
        {"name": "pcg_small8_fp64", "kind": "pcg", "geometry": "small", "natoms": 8, "nchi": 4, "k": 1, "steps": 10,
         "precision": "fp64", "precond": "iter"},
        # FP64 at the size where arithmetic counts: a reference run that mixed precision is checked against
        {"name": "apply_cluster32_fp64", "kind": "apply", "geometry": "cluster", "natoms": 32, "nchi": 9, "k": 3,
         "precision": "fp64"},
        # the smallest system of a batch of uneven ones, two states: latency in mixed precision
        {"name": "apply_cluster20_mixed", "kind": "apply", "geometry": "cluster", "natoms": 20, "nchi": 4, "k": 2,
         "precision": "mixed"},
        # the benchmark's operator: 140 atoms with 4 + 9 functions each, ten states
        {"name": "apply_chromo140_mixed", "kind": "apply", "geometry": "chromophore", "natoms": 140, "nchi": 9, "k": 10,
         "precision": "mixed"},
        # the benchmark's solver: truncated response kernels, the exact preconditioner
        {"name": "pcg_chromo140_exact", "kind": "pcg", "geometry": "chromophore", "natoms": 140, "nchi": 9, "k": 10,
         "steps": 2, "precision": "mixed", "precond": "exact"},
        # a mid-size system of a batch with the paper's inner CG as preconditioner
        {"name": "pcg_cluster60_iter", "kind": "pcg", "geometry": "cluster", "natoms": 60, "nchi": 4, "k": 5, "steps": 2,
         "precision": "mixed", "precond": "iter"},
        # the large end of a batch: condensed-phase density, tiles denser than one unit; odd state count
        {"name": "density_cluster200", "kind": "density", "geometry": "cluster", "natoms": 200, "nchi": 4, "k": 5,
         "precision": "mixed"},
        # the other direction of the grid work, at the chromophore's tile shapes; odd state count
        {"name": "integrals_chromo140", "kind": "integrals", "geometry": "chromophore", "natoms": 140, "nchi": 9, "k": 7,
         "precision": "mixed"},
        # Hartree and exchange-correlation potential on the 0.25 A grid of a 36 A cell
        {"name": "potential_144", "kind": "potential", "geometry": "grid", "natoms": 4, "nchi": 4, "grid": 144, "k": 8,
         "precision": "mixed"},
        # the truncated (linear-scaling) form on a core in its solvent shell
        {"name": "apply_shell200_sparse", "kind": "apply", "geometry": "shell", "natoms": 200, "nchi": 9, "k": 4,
         "precision": "mixed"},
        # training and inference of the learned preconditioner at its default width
        {"name": "mlp_16384", "kind": "mlp", "rows": 16384, "width": 256, "n_block": 32, "n_feat": 65},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply64", "pcg64", "apply", "apply", "pcg", "density", "integrals", "potential", "sparse", "mlp"])
    if kind == "apply64":
        g = rng.choice(["small", "cluster"])
        return {"kind": "apply", "geometry": g, "natoms": _log_int(rng, 8, 30), "nchi": rng.choice([4, 9]),
                "k": rng.randint(1, 3), "precision": "fp64"}
    if kind == "pcg64":
        return {"kind": "pcg", "geometry": "small", "natoms": _log_int(rng, 8, 20), "nchi": 4, "k": rng.randint(1, 3),
                "steps": rng.randint(2, 10), "precision": "fp64", "precond": "iter"}
    if kind == "pcg":
        return {"kind": "pcg", "geometry": "cluster", "natoms": _log_int(rng, 20, 60), "nchi": 4, "k": rng.randint(1, 8),
                "steps": 2, "precision": "mixed", "precond": rng.choice(["iter", "exact"])}
    if kind in ("apply", "density", "integrals"):
        g = rng.choice(["chromophore", "cluster"])
        natoms = _log_int(rng, 40, 140) if g == "chromophore" else _log_int(rng, 20, 200)
        nchi = rng.choice([4, 9]) if natoms <= 140 else 4
        return {"kind": kind, "geometry": g, "natoms": natoms, "nchi": nchi,
                "k": rng.randint(1, 10 if g == "chromophore" else 5), "precision": "mixed"}
    if kind == "potential":
        return {"kind": "potential", "geometry": "grid", "natoms": 4, "nchi": 4,
                "grid": synthetic.smooth_grid(rng.randint(40, 150)), "k": rng.randint(1, 10),
                "precision": rng.choice(["mixed", "mixed", "fp64"])}
    if kind == "sparse":
        return {"kind": "apply", "geometry": "shell", "natoms": _log_int(rng, 60, 180), "nchi": 9, "k": rng.randint(1, 4),
                "precision": "mixed"}
    return {"kind": "mlp", "rows": _log_int(rng, 300, 16384), "width": rng.choice([64, 128, 256]),
            "n_block": 32, "n_feat": 65}


# ---- systems and contexts -----------------------------------------------------------------------

def _recipe(case):
    g, na = case["geometry"], case["natoms"]
    if g == "small":          # the smallest workload's density: 1/3 A grid, 7 A functions, whole cell
        return dataclasses.replace(synthetic.small_density_recipe(na, 1), nchi=case["nchi"])
    if g == "chromophore":    # the chromophore workload in a cell of twice its functions' boxes (0.25 A grid)
        n = synthetic.smooth_grid(int(math.ceil(135.0 * max(1.0, na / 140.0) ** (1.0 / 3.0))))
        return dataclasses.replace(synthetic.CONFIG_CHROMOPHORE, natoms=na, nchi=case["nchi"], ngrid=n, cell_ang=0.25 * n,
                                   fast=True)
    if g == "cluster":        # a system of the uneven batches: 0.1 atoms / A^3 in vacuum, 7 A functions; 0.25 A
        side, radius, h = (na / 0.1) ** (1.0 / 3.0), 7.0, 0.25                 # grid, smaller ones 1/3 A
        n = synthetic.smooth_grid(int(math.ceil((side + 2.0 * radius + 1.0) / h)))
        if n < 120:
            h, n = 1.0 / 3.0, 90
        return synthetic.Recipe(natoms=na, cell_ang=n * h, ngrid=n, nchi=case["nchi"], radius_ang=radius,
                                cluster_ang=side, seed=7000 + na, fast=True)
    if g == "shell":          # the linear-scaling series' recipe
        return dataclasses.replace(synthetic.scaling_recipe(na), nchi=case["nchi"])
    n = case["grid"]          # a few small functions: only the grid matters
    return synthetic.Recipe(natoms=case["natoms"], cell_ang=0.25 * n, ngrid=n, nchi=case["nchi"], radius_ang=3.0, seed=3)


@functools.lru_cache(maxsize=2)
def _system_of(key):
    return synthetic.generate(_recipe(dict(key)))


def _system(case):
    return _system_of(tuple(sorted((k, case[k]) for k in ("geometry", "natoms", "nchi", "grid") if k in case)))


@functools.lru_cache(maxsize=1)
def _context_of(key):
    case = dict(key)
    # a context makes the exact preconditioner's bases only when asked for it
    return tddft.Context(_system(case), sparse=case["geometry"] == "shell", precision=case["precision"],
                         precond=case.get("precond", "none" if case["geometry"] == "shell" else "iter"))


def _context(case):
    keys = ("geometry", "natoms", "nchi", "grid", "precision", "precond")
    return _context_of(tuple(sorted((k, case[k]) for k in keys if k in case)))


# ---- inputs ---------------------------------------------------------------------------------------

def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _randn(seed, salt, *shape):
    return torch.randn(*shape, generator=_gen(seed, salt), device=DEV, dtype=torch.float64)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV, torch.float64)


def _atom_mask(s):
    """[natoms][natoms] of atom pairs within the kernel cutoff (minimum image)."""
    d = s.pos[:, None, :] - s.pos[None, :, :]
    d -= s.cell * np.rint(d / s.cell)
    return torch.from_numpy(np.sqrt((d * d).sum(-1)) <= s.kernel_cutoff).to(DEV)


def _to_blocks(s, x):
    """[k][N_chi][N_phi] -> [k][nnz]: the atom blocks within the cutoff, row-major (the sparse boundary)."""
    k, na, nc, nv = x.shape[0], s.natoms, s.recipe.nchi, s.recipe.nphi
    b = x.reshape(k, na, nc, na, nv).permute(0, 1, 3, 2, 4)
    return b[:, _atom_mask(s)].reshape(k, -1).contiguous()


def _from_blocks(s, x):
    k, na, nc, nv = x.shape[0], s.natoms, s.recipe.nchi, s.recipe.nphi
    b = torch.zeros(k, na, na, nc, nv, dtype=x.dtype, device=x.device)
    b[:, _atom_mask(s)] = x.reshape(k, -1, nc, nv)
    return b.permute(0, 1, 3, 2, 4).reshape(k, na * nc, na * nv)


def _kernels(s, k, seed, salt):
    """Response kernels as the solver holds them: P^c S^chi L S^phi P^v of random L, unit scale."""
    L = _randn(seed, salt, k, s.chi.nfun, s.phi.nfun)
    P = (_dev(s.P_c) @ _dev(s.S_chi)) @ L @ (_dev(s.S_phi) @ _dev(s.P_v))
    return (P / P.square().mean(dim=(1, 2), keepdim=True).sqrt()).contiguous()


def _fields(n, k, seed, salt):
    """Smooth periodic fields of zero mean: a few long waves and a little noise."""
    x = torch.arange(n, device=DEV, dtype=torch.float64) * (2.0 * math.pi / n)
    out = 0.01 * _randn(seed, salt, k, n, n, n)
    w = _randn(seed, salt + 1, k, 6, 5).cpu()
    for s in range(k):
        for q in range(6):
            m = [1 + (q + a) % 3 for a in range(3)]
            a, b, c = (torch.cos(m[i] * x + float(w[s, q, i])) for i in range(3))
            out[s] += float(w[s, q, 3]) * a[:, None, None] * b[None, :, None] * c[None, None, :]
    return 0.1 * (out - out.mean(dim=(1, 2, 3), keepdim=True))


def _mlp_inputs(case, seed):
    g = _gen(seed, 5)
    n, nb, nf = case["rows"], case["n_block"], case["n_feat"]
    X = torch.randn(n, nb + nf, generator=g, device=DEV)
    X[:, :nb] /= X[:, :nb].norm(dim=1, keepdim=True)
    T = 0.3 * torch.randn(n, nb, generator=g, device=DEV) / math.sqrt(nb)
    w = torch.rand(n, generator=g, device=DEV) ** 4
    return X, T, w / w.sum(), synthetic.mlp_init(nf, case["width"], nb * nb, int(seed))


def prepare(case, seed):
    if case["kind"] == "mlp":
        X, T, w, theta = _mlp_inputs(case, seed)
        mlp = tddft.Mlp(case["n_block"], case["n_feat"], case["width"])
        mlp.set(theta)
        return {"case": case, "mlp": mlp, "X": X, "T": T, "w": w}
    s, ctx, k = _system(case), _context(case), case["k"]
    st = {"case": case, "ctx": ctx, "lib": tddft.load()}
    if case["kind"] == "apply":
        P = [_kernels(s, k, seed, salt) for salt in (1, 2)]
        if case["geometry"] == "shell":
            P = [_to_blocks(s, p) for p in P]
        st["in"] = P
        st["out"] = [torch.empty_like(p) for p in P]
    elif case["kind"] == "pcg":
        st["in"] = [_randn(seed, 1, k, s.chi.nfun, s.phi.nfun)]
        st["out"] = [torch.empty_like(st["in"][0]) for _ in range(6)]
    elif case["kind"] == "density":
        st["in"] = [_kernels(s, k, seed, 1)]
    else:
        st["in"] = [_fields(s.n, k, seed, 1)]
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "mlp":
        loss, grad = st["mlp"].loss_grad(st["X"], st["T"], st["w"])
        return loss, grad, st["mlp"].forward(st["X"])
    ctx = st["ctx"]
    if kind == "apply":
        out = list(ctx.apply(*st["in"], *st["out"]))
    elif kind == "density":
        out = [ctx.response_density(st["in"][0])]
    elif kind == "potential":
        out = [ctx.response_potential(st["in"][0])]
    elif kind == "integrals":
        out = [ctx.potential_integrals(st["in"][0])]
    else:
        s = ctx.state(st["in"][0])
        for _ in range(case["steps"]):
            om, res = s.step()
        # the new iterate, into the program's own buffers: P, f and L of both halves
        ctx._check(st["lib"].tddft_state_get(ctx._ctx, s._st, *(x.data_ptr() for x in st["out"])))
        s.close()
        out = [torch.from_numpy(om), torch.from_numpy(res), *st["out"]]
    return out if case["precision"] == "fp64" else [x.float() for x in out]


# ---- work -----------------------------------------------------------------------------------------

def _lens_points(s):
    """(sum over (chi, phi) pairs of the grid points both cover, grid points of all functions)."""
    R = s.recipe.radius_ang * synthetic.BOHR_PER_ANG
    d = s.pos[:, None, :] - s.pos[None, :, :]
    d -= s.cell * np.rint(d / s.cell)
    d = np.minimum(np.sqrt((d * d).sum(-1)), 2.0 * R)
    lens = (math.pi * (4.0 * R + d) * (2.0 * R - d) ** 2 / 12.0).sum() / s.dV
    ball = 4.0 / 3.0 * math.pi * R ** 3 / s.dV
    r = s.recipe
    return float(lens) * r.nchi * r.nphi, ball * s.natoms * (r.nchi + r.nphi)


def work(case):
    if case["kind"] == "mlp":
        n, w, nb, nf = case["rows"], case["width"], case["n_block"], case["n_feat"]
        size = nf * w + w + w * w + w + w * nb * nb + nb * nb
        gemm = 2.0 * n * (nf * w + w * w + w * nb * nb)
        # loss and gradient: forward, dW and dH of each layer (no dX of the first); and one more forward
        flops = 4.0 * gemm - 2.0 * n * nf * w + 6.0 * n * nb * nb
        return {"bytes": 4.0 * (n * (nb + nf) + n * nb + n + 2 * size + n * nb), "flops": flops}
    s, k = _system(case), case["k"]
    el = 8.0 if case["precision"] == "fp64" else 4.0
    nc, nv, n3 = s.chi.nfun, s.phi.nfun, float(s.n) ** 3
    pairs, table = _lens_points(s)
    grid = 2.0 * k * pairs
    fft = 2.0 * 5.0 * n3 * math.log2(n3) * ((k + 1) // 2)
    if case["kind"] == "potential":
        return {"bytes": 2 * 8.0 * k * n3 + el * n3, "flops": fft}
    if case["kind"] in ("density", "integrals"):
        return {"bytes": el * table + 8.0 * k * (n3 + nc * nv), "flops": grid}
    left, right = 2.0 * nc * nc * nv, 2.0 * nc * nv * nv
    fill = 1.0
    if case["geometry"] == "shell":
        fill = float(_atom_mask(s).double().mean())
        left, right = left * fill * fill, right * fill * fill
    consts = 2.0 * fill * (nc * nc + nv * nv)
    once = {"bytes": 8.0 * 4 * k * fill * nc * nv + el * (table + consts + n3), "flops": 3 * k * (left + right) + 2 * grid + fft}
    if case["kind"] == "apply":
        return once
    # a step: one application, and per matrix of the 2 k the products of cov(g), the preconditioner,
    # Eq. auxiliary and cov(D); the start adds one application and two maps
    steps = case["steps"]
    per = once["flops"] + 2 * k * 4 * (left + right) + 2 * k * 2 * k * 6 * 2.0 * nc * nv
    vec = el * 2 * k * nc * nv
    return {"bytes": 8.0 * 7 * k * nc * nv + (steps + 1) * (el * (table + 3 * consts + n3) + 8 * vec),
            "flops": steps * per + once["flops"] + 2 * k * 2 * (left + right)}


# ---- the same in 64 bits ---------------------------------------------------------------------------

def _full_tables(fs, nper, n):
    """Every function on the whole grid [nfun][n][n][n], in the tables' own type."""
    e = int(fs.box[0, 3])
    val = torch.from_numpy(fs.val).to(DEV).reshape(-1, nper, e, e, e)
    full = torch.zeros(fs.nfun, n, n, n, dtype=val.dtype, device=DEV)
    t = torch.arange(e, device=DEV)
    for a in range(val.shape[0]):
        ix, iy, iz = ((int(o) + t) % n for o in fs.box[a * nper, :3])
        full[a * nper:(a + 1) * nper, ix[:, None, None], iy[None, :, None], iz[None, None, :]] = val[a]
    return full


def _touching(fs, n, lo, hi):
    """Functions whose box meets the block of points [lo, hi) of every axis."""
    ok = np.ones(fs.nfun, dtype=bool)
    for a in range(3):
        o, e = fs.box[:, a].astype(np.int64), fs.box[:, 3 + a].astype(np.int64)
        ok &= ((lo[a] - o) % n < e) | ((o - lo[a]) % n < hi[a] - lo[a])
    return torch.from_numpy(np.nonzero(ok)[0]).to(DEV)


def _blocks(s):
    """For blocks of the grid: (slices, chi ids, phi ids, chi values, phi values [functions][points])."""
    n, B, r = s.n, 12, s.recipe
    chi, phi = _full_tables(s.chi, r.nchi, n), _full_tables(s.phi, r.nphi, n)
    for x in range(0, n, B):
        for y in range(0, n, B):
            for z in range(0, n, B):
                lo, hi = (x, y, z), (min(x + B, n), min(y + B, n), min(z + B, n))
                ic, ip = _touching(s.chi, n, lo, hi), _touching(s.phi, n, lo, hi)
                if len(ic) and len(ip):
                    sl = tuple(slice(a, b) for a, b in zip(lo, hi))
                    yield (sl, ic, ip, chi[(ic, *sl)].double().reshape(len(ic), -1),
                           phi[(ip, *sl)].double().reshape(len(ip), -1))


def _exact_density(s, P):
    rho = torch.zeros(P.shape[0], s.n, s.n, s.n, dtype=torch.float64, device=DEV)
    for sl, ic, ip, c, p in _blocks(s):
        t = torch.matmul(c.T, P[:, ic[:, None], ip])                       # [k][points][phi]
        d = torch.einsum("krb,br->kr", t, p)
        rho[(slice(None), *sl)] = d.reshape(-1, *(q.stop - q.start for q in sl))
    return rho


def _exact_fxc(s):
    n0 = _dev(s.n0)
    n = n0.clamp_min(1e-10).requires_grad_(True)
    rs = (3.0 / (4.0 * math.pi * n)) ** (1.0 / 3.0)
    q = rs.sqrt()
    ec = -2 * 0.031091 * (1 + 0.21370 * rs) * torch.log1p(
        1.0 / (2 * 0.031091 * (7.5957 * q + 3.5876 * rs + 1.6382 * q * rs + 0.49294 * rs * rs)))
    e = n * (ec - 0.75 * (3.0 / math.pi) ** (1.0 / 3.0) * n ** (1.0 / 3.0))
    (g,) = torch.autograd.grad(e.sum(), n, create_graph=True)
    (f,) = torch.autograd.grad(g.sum(), n)
    return torch.where(n0 >= 1e-10, f, torch.zeros_like(f)).detach()


def _exact_potential(s, rho):
    m = torch.fft.fftfreq(s.n, 1.0 / s.n, device=DEV, dtype=torch.float64) * (2.0 * math.pi / s.cell)
    g2 = m[:, None, None] ** 2 + m[None, :, None] ** 2 + m[None, None, :] ** 2
    g2[0, 0, 0] = 1.0
    kern = 4.0 * math.pi / g2
    kern[0, 0, 0] = 0.0
    f = _exact_fxc(s)
    return torch.stack([torch.fft.ifftn(torch.fft.fftn(r) * kern).real + f * r for r in rho])


def _exact_integrals(s, V):
    out = torch.zeros(V.shape[0], s.chi.nfun, s.phi.nfun, dtype=torch.float64, device=DEV)
    for sl, ic, ip, c, p in _blocks(s):
        v = V[(slice(None), *sl)].reshape(V.shape[0], 1, -1)
        out[:, ic[:, None], ip] += torch.matmul(c * v, p.T)
    return out * s.dV


def exact(case, seed):
    kind = case["kind"]
    if kind == "pcg":
        return None     # the iterates depend on the solver's own decisions (line search, inner stops)
    if kind == "mlp":
        X, T, w, theta = _mlp_inputs(case, seed)
        nb, nf, wd = case["n_block"], case["n_feat"], case["width"]
        sizes = [(nf, wd), (wd,), (wd, wd), (wd,), (wd, nb * nb), (nb * nb,)]

        def split(t):
            parts, o = [], 0
            for sh in sizes:
                m = math.prod(sh)
                parts.append(t[o:o + m].reshape(sh))
                o += m
            return parts

        def model(t):
            W1, b1, W2, b2, W3, b3 = split(t)
            h = torch.relu(X[:, nb:].double() @ W1 + b1)
            A = (torch.relu(h @ W2 + b2) @ W3 + b3).reshape(-1, nb, nb)
            return torch.einsum("rij,rj->ri", A, X[:, :nb].double())

        th = torch.from_numpy(theta).to(DEV)
        t64 = th.double().requires_grad_(True)
        loss = (w.double()[:, None] * (model(t64) - T.double()) ** 2).sum() / (X.shape[0] * nb)
        (g,) = torch.autograd.grad(loss, t64)
        with torch.no_grad():
            y = model(th.bfloat16().double())
        return float(loss), g.cpu().numpy(), y
    s, k = _system(case), case["k"]
    if kind == "density":
        return [_exact_density(s, _kernels(s, k, seed, 1))]
    if kind == "potential":
        return [_exact_potential(s, _fields(s.n, k, seed, 1))]
    if kind == "integrals":
        return [_exact_integrals(s, _fields(s.n, k, seed, 1))]
    P = [_kernels(s, k, seed, salt) for salt in (1, 2)]
    Pc, Pv, Hc, Hv = _dev(s.P_c), _dev(s.P_v), _dev(s.H_chi), _dev(s.H_phi)

    def cut(x):
        return x

    if case["geometry"] == "shell":
        keep = _atom_mask(s)                     # both cutoffs of the series are equal
        nc, nv = s.recipe.nchi, s.recipe.nphi
        Pc = Pc * keep.repeat_interleave(nc, 0).repeat_interleave(nc, 1)
        Pv = Pv * keep.repeat_interleave(nv, 0).repeat_interleave(nv, 1)
        m = keep.repeat_interleave(nc, 0).repeat_interleave(nv, 1)

        def cut(x):
            return x * m

        P = [cut(p) for p in P]
    Mc, Mv = Pc @ Hc, Hv @ Pv
    fp, fq = (cut(Mc @ p) - cut(p @ Mv) for p in P)
    V = cut(_exact_integrals(s, _exact_potential(s, _exact_density(s, P[1]))))
    fq = fq + 2.0 * cut(cut(Pc @ V) @ Pv)
    return [_to_blocks(s, f) for f in (fp, fq)] if case["geometry"] == "shell" else [fp, fq]
