"""What a program built on this framework has it do, as cases that can be timed.

A case is a dict of plain values: the kind of call, the lattice, the number of
moments, the precision.  listed() holds the fixed cases, draw() gives more of
the same ranges, prepare() makes what a program has in hand before the call,
run() is one pass through the public entry points, work() counts what the
pass cannot do without and exact() computes the same outputs in 64 bits with
plain torch.

Sizes follow this repository's own workloads (the 16 x 16 clean lattice, the
128 x 128 disordered one, the d-wave vortex lattice, the ensemble of uneven
disorder realisations, the 64 x 64 gradient, the S/N slab and the S/N/S
junction), at sizes a pass of which takes at most a few tenths of a second.

A lattice built with the FP32 recursion promises single precision (moments to
1e-5, Delta to 1e-4), so the program keeps what it returns as float32 or
complex64; results of the FP64 recursion stay in 64 bits.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1007_1609_gb300 import cbdg

DX = (1, -1, 0, 0, 1, -1, 1, -1)
DY = (0, 0, 1, -1, 1, -1, -1, 1)


def listed():
    return [
        # The smallest whole program: ten mixed self-consistency iterations of
        # the clean 16 x 16 lattice in FP64, where launches and latency count.
        dict(name="scf_16x16_fp64", kind="scf", lx=16, ly=16, px=0, py=0, M=256, precision="fp64", W=0.0, iters=10),
        # A small ragged disordered lattice in FP32, a few iterations: what a
        # parameter scan over many small samples does.
        dict(name="scf_33x21_fp32", kind="scf", lx=33, ly=21, px=0, py=0, M=512, precision="fp32", W=1.0, iters=4),
        # The FP64 form of the disordered lattice at a size where the vectors
        # no longer fit on chip: the reference run beside an FP32 one.
        dict(name="map_61x45_fp64", kind="map", lx=61, ly=45, px=0, py=0, M=512, precision="fp64", W=1.0),
        # One self-consistency map of the 128 x 128 disordered lattice, every
        # site a start vector: the headline workload.
        dict(name="map_128x128_fp32", kind="map", lx=128, ly=128, px=0, py=0, M=1024, precision="fp32", W=1.0),
        # The same map on a torus of odd sides (bulk averages over disorder
        # without surfaces).
        dict(name="map_torus_75x90_fp32", kind="map", lx=75, ly=90, px=1, py=1, M=512, precision="fp32", W=1.0),
        # Local density of states at a handful of sites around an impurity of
        # the S/N/S junction: few start vectors, many moments.
        dict(name="ldos_junction_100x150", kind="ldos", lx=100, ly=150, px=0, py=0, M=2048, precision="fp32", sites=11,
             energies=201),
        # The planar S/N slab with one start vector per layer: a wide lattice
        # with few columns, one self-consistency map with per-site couplings.
        dict(name="map_slab_500x320", kind="slab", lx=500, ly=320, px=1, py=0, M=1024, precision="fp32"),
        # LDOS map of a patch of the d-wave vortex lattice (complex vectors,
        # t', bond pairing, field): recursion and dense contraction.
        dict(name="ldos_vortex_96x96", kind="vortex_ldos", lx=96, ly=96, px=1, py=1, M=1024, precision="fp32", sites=512,
             energies=512),
        # Bond currents of a vortex lattice: every site a complex start vector.
        dict(name="currents_vortex_64x64", kind="currents", lx=64, ly=64, px=1, py=1, M=512, precision="fp32"),
        # Nonlocal Green's functions between a few sites and a patch around a
        # vortex core, left on the GPU.
        dict(name="green_vortex_128x128", kind="green", lx=128, ly=128, px=1, py=1, M=1024, precision="fp32", sites=16,
             targets=256, energies=512),
        # One iteration of an ensemble of uneven disorder realisations.
        dict(name="ensemble_16", kind="ensemble", members=16, lo=32, hi=96, M=512, precision="fp32"),
        # Gradient of a loss on Delta with respect to every parameter (reverse
        # mode), the 64 x 64 workload.
        dict(name="grad_64x64_fp32", kind="grad", lx=64, ly=64, px=0, py=0, M=512, precision="fp32", W=1.0),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    # (the torus, the FP64 map and the disordered one are one kind: "map")
    kind = rng.choice(["scf", "map", "map", "map", "ldos", "slab", "vortex_ldos", "currents", "green", "ensemble",
                       "grad"])
    per = rng.choice([(0, 0), (0, 0), (1, 1), (1, 0), (0, 1)])
    if kind == "scf":
        precision = rng.choice(["fp32", "fp64"])
        top = 48 if precision == "fp32" else 24
        return dict(kind=kind, lx=log(6, top), ly=log(6, top), px=0, py=0, M=log(64, 512), precision=precision,
                    W=rng.choice([0.0, 1.0]), iters=rng.randint(2, 8))
    if kind == "map":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        while True:
            c = dict(kind=kind, lx=log(8, 128), ly=log(8, 128), px=per[0], py=per[1], M=log(128, 1024),
                     precision=precision, W=rng.choice([0.5, 1.0, 2.0]))
            if (c["lx"] * c["ly"]) ** 2 * c["M"] <= 128 ** 4 * 1024 / (64 if precision == "fp64" else 1 + per[1]):
                return c
    if kind == "ldos":
        return dict(kind=kind, lx=log(40, 200), ly=log(60, 240), px=0, py=0, M=log(256, 2048), precision="fp32",
                    sites=log(1, 64), energies=log(51, 501))
    if kind == "slab":
        return dict(kind=kind, lx=log(64, 500), ly=log(64, 320), px=1, py=0, M=log(256, 1024), precision="fp32")
    if kind == "vortex_ldos":
        return dict(kind=kind, lx=log(24, 96), ly=log(24, 96), px=1, py=1, M=log(128, 1024), precision="fp32",
                    sites=log(32, 512), energies=log(64, 512))
    if kind == "currents":
        return dict(kind=kind, lx=log(16, 64), ly=log(16, 64), px=1, py=1, M=log(64, 512), precision="fp32")
    if kind == "green":
        return dict(kind=kind, lx=log(32, 128), ly=log(32, 128), px=1, py=1, M=log(128, 1024), precision="fp32",
                    sites=log(1, 16), targets=log(16, 256), energies=log(64, 512))
    if kind == "ensemble":
        return dict(kind=kind, members=log(4, 16), lo=rng.choice([24, 32]), hi=rng.choice([64, 80, 96]),
                    M=log(128, 512), precision="fp32")
    return dict(kind=kind, lx=log(16, 64), ly=log(16, 64), px=per[0], py=per[1], M=log(64, 512), precision="fp32",
                W=rng.choice([0.5, 1.0]))


# ------------------------------------------------------------------ inputs


def _neighbours(lx, ly, px, py, nd):
    """[N, nd] neighbour site along each direction, -1 across an open edge."""
    s = np.arange(lx * ly)
    x, y = s % lx, s // lx
    out = np.empty((s.size, nd), dtype=np.int64)
    for d in range(nd):
        nx, ny = x + DX[d], y + DY[d]
        cut = np.zeros(s.size, dtype=bool)
        if not px:
            cut |= (nx < 0) | (nx >= lx)
        if not py:
            cut |= (ny < 0) | (ny >= ly)
        out[:, d] = np.where(cut, -1, nx % lx + lx * (ny % ly))
    return out


def _hops(lx, ly, px, py, t=1.0, tp=0.0, flux=0.0):
    """t_ij of every directed bond; flux h/2e quanta through the periodic cell
    (Landau gauge A = (0, B x), twist on the bonds across the x seam)."""
    nd = 8 if tp else 4
    nb = _neighbours(lx, ly, px, py, nd)
    s = np.arange(lx * ly)
    x, y = s % lx, s // lx
    hop = np.zeros((s.size, nd), dtype=np.complex128)
    phi, twist = math.pi * flux / (lx * ly), math.pi * flux / ly
    for d in range(0, nd, 2):
        on = nb[:, d] >= 0
        theta = phi * (x + 0.5 * DX[d]) * DY[d]
        seam = (x + DX[d] < 0) | (x + DX[d] >= lx)
        theta = theta - np.where(seam, twist * ((y + DY[d]) % ly), 0.0)
        val = (t if d < 4 else tp) * np.exp(1j * theta)
        hop[on, d] = val[on]
        hop[nb[on, d], d + 1] = np.conj(val[on])
    return hop


def _onsite(lx, ly, px, py, W, rng, mu=-0.5, U=2.0, T=0.01):
    """Disordered s-wave lattice; Delta near 0.5, as after a few iterations."""
    n = lx * ly
    eps = rng.uniform(-0.5 * W, 0.5 * W, n) if W else np.zeros(n)
    delta = 0.5 * (1.0 + 0.1 * rng.standard_normal(n).clip(-3, 3)).astype(np.complex128)
    return SimpleNamespace(Lx=lx, Ly=ly, periodic_x=px, periodic_y=py, eps=eps, mu=mu, hop=_hops(lx, ly, px, py),
                           pairing=cbdg.CBDG_ONSITE_U, coupling=U, delta0=delta, T=T)


def _dwave(lx, ly, rng):
    """d-wave vortex lattice: t' = -0.3, two h/2e quanta, two vortices on the
    diagonal in the bond Delta, weak disorder."""
    n = lx * ly
    nb = _neighbours(lx, ly, 1, 1, 4)
    s = np.arange(n)
    x, y = s % lx, s // lx
    shift = rng.uniform(0.2, 0.8, 2)
    delta = np.zeros((n, 4), dtype=np.complex128)
    for d in (0, 2):
        mx, my = x + 0.5 * DX[d], y + 0.5 * DY[d]
        z = np.full(n, 0.5 if d == 0 else -0.5, dtype=np.complex128)
        for k in range(2):
            rx, ry = mx - (k + 0.5) * lx / 2 - shift[0], my - (k + 0.5) * ly / 2 - shift[1]
            z = z * np.tanh(np.hypot(rx, ry) / 3.0) * np.exp(1j * np.arctan2(ry, rx))
        delta[s, d] = z
        delta[nb[:, d], d + 1] = z
    return SimpleNamespace(Lx=lx, Ly=ly, periodic_x=1, periodic_y=1, eps=rng.uniform(-0.1, 0.1, n), mu=-1.0,
                           hop=_hops(lx, ly, 1, 1, tp=-0.3, flux=2.0), pairing=cbdg.CBDG_BOND_V, coupling=1.5,
                           delta0=delta, T=0.005)


def _problem(case, seed):
    """Everything of the case that is plain numbers, from the seed alone."""
    rng = np.random.Generator(np.random.PCG64(seed))
    kind = case["kind"]
    if kind == "ensemble":
        # the members' sides go with the case, their disorder with the seed
        sizes = np.random.Generator(np.random.PCG64(1003 + case["members"]))
        sides = sizes.integers(case["lo"] // 8, case["hi"] // 8 + 1, case["members"]) * 8
        sides[0], sides[-1] = case["lo"], case["hi"]
        return [_onsite(int(L), int(L), 0, 0, rng.uniform(0.5, 2.0), rng) for L in sides]
    lx, ly = case["lx"], case["ly"]
    n = lx * ly
    if kind in ("scf", "map"):
        return _onsite(lx, ly, case["px"], case["py"], case["W"], rng)
    if kind == "ldos":
        # junction: a third of the layers normal, a Gaussian impurity in them
        p = _onsite(lx, ly, 0, 0, 0.0, rng, U=1.41, T=0.005)
        x, y = np.arange(n) % lx, np.arange(n) // lx
        x0, y0 = int(rng.integers(lx // 3, lx - lx // 3)), int(rng.integers(ly // 3, ly - ly // 3))
        p.eps = 2.0 * np.exp(-((x - x0) ** 2 + (y - y0) ** 2).astype(np.float64))
        p.delta0 = np.where((y < ly // 3) | (y >= ly - ly // 3), 0.1, 0.0) + 0.01 * p.delta0
        near = np.argsort((x - x0) ** 2 + (y - y0) ** 2, kind="stable")
        p.sites = near[:case["sites"]].astype(np.int32)
        p.energies = np.linspace(-0.35, 0.35, case["energies"])
        return p
    if kind == "slab":
        # translation invariant along x: one start vector per layer
        p = _onsite(lx, ly, 1, 0, 0.0, rng, U=1.41, T=0.005)
        y = np.arange(n) // lx
        layer = 0.1 * (1.0 + 0.1 * rng.standard_normal(ly).clip(-3, 3))
        p.n_s = ly - max(1, ly // 16)
        p.U_site = np.where(y < p.n_s, 1.41, 0.0)
        p.delta0 = np.where(y < p.n_s, layer[y], 0.1 * layer[y]).astype(np.complex128)
        p.rep = (lx * y).astype(np.int32)
        return p
    if kind == "grad":
        p = _onsite(lx, ly, case["px"], case["py"], case["W"], rng)
        x, y = np.arange(n) % lx, np.arange(n) // lx
        bump = np.exp(-((x - 0.5 * (lx - 1)) ** 2 + (y - 0.5 * (ly - 1)) ** 2) / 128.0)
        # dL/dDelta_out of L = sum (Delta - target)^2 at a Delta near the input
        p.weight = (2.0 * (p.delta0 - (0.4 + 0.3 * bump))).astype(np.complex128)
        return p
    p = _dwave(lx, ly, rng)
    if kind == "vortex_ldos":
        p.sites = rng.permutation(n)[:min(n, case["sites"])].astype(np.int32)
        p.energies = np.linspace(-4.0, 4.0, case["energies"])
    if kind == "green":
        x, y = np.arange(n) % lx, np.arange(n) // lx
        near = np.argsort((x - lx // 4) ** 2 + (y - ly // 4) ** 2, kind="stable")
        p.sites = near[:min(n, case["sites"])].astype(np.int32)
        p.targets = near[:min(n, case["targets"])].astype(np.int32)
        p.energies = np.linspace(-3.0, 3.0, case["energies"])
    return p


def prepare(case, seed):
    p = _problem(case, seed)
    if case["kind"] == "ensemble":
        return SimpleNamespace(case=case, p=p, ens=cbdg.Ensemble(p))
    lat = cbdg.Lattice(p, precision=case["precision"])
    st = SimpleNamespace(case=case, p=p, lat=lat)
    if case["kind"] == "slab":
        lat.set_coupling(p.U_site)
        lat.set_symmetry(p.rep)
    if case["kind"] == "green":
        shape = (p.sites.size, p.targets.size, p.energies.size)
        st.g = [torch.empty(shape, dtype=torch.complex128, device="cuda") for _ in range(2)]
        st.e = torch.from_numpy(p.energies).cuda()
    return st


# --------------------------------------------------------------------- pass


def _kept(case, x):
    """Results of the FP32 recursion in single precision, of FP64 as they are."""
    if case["precision"] == "fp64":
        return x
    return x.astype(np.complex64 if np.iscomplexobj(x) else np.float32)


def run(st):
    c, kind = st.case, st.case["kind"]
    if kind == "ensemble":
        st.ens.scf(0.01, c["M"], 0.5, 0.0, 1)
        return [_kept(c, st.ens.delta(k)) for k in range(c["members"])]
    p, lat, M = st.p, st.lat, c["M"]
    if kind == "scf":
        lat.delta = p.delta0
        moved = [lat.scf_step(p.T, M, 0.5) for _ in range(c["iters"])]
        return {"delta": _kept(c, lat.delta), "moved": _kept(c, np.array(moved))}
    if kind in ("map", "slab"):
        delta, n = lat.order_parameter(p.T, M)
        return {"delta": _kept(c, delta), "n": _kept(c, n)}
    if kind == "ldos":
        lam = lat.lorentz_lambda(0.01, M)
        return lat.ldos(p.sites, M, p.energies, kernel="lorentz", lam=lam)
    if kind == "vortex_ldos":
        return lat.ldos(p.sites, M, p.energies)
    if kind == "currents":
        return _kept(c, lat.bond_currents(p.T, M))
    if kind == "green":
        cbdg.cbdg_green_function(lat.handle, p.sites, p.sites.size, p.targets, p.targets.size, M, cbdg.CBDG_JACKSON,
                                 0.0, st.e, p.energies.size, st.g[0], st.g[1])
        return [g.to(torch.complex64) for g in st.g]
    g_eps, g_hop, g_delta = lat.backward(p.T, M, p.weight)
    return {"eps": _kept(c, g_eps), "hop": _kept(c, g_hop), "delta": _kept(c, g_delta)}


def _columns(case):
    if case["kind"] == "slab":
        return case["ly"]
    n = case["lx"] * case["ly"]
    return min(n, case["sites"]) if "sites" in case else n


def work(case):
    """Inputs read once and outputs written once; the recursion's multiply-adds:
    per site and step 12 of the real stencil and 6 of the column products (two
    moments a step), 112 of the complex stencil (one moment a step)."""
    kind, M = case["kind"], case["M"]
    if kind == "ensemble":
        n2 = n = 0
        for L in np.linspace(case["lo"], case["hi"], case["members"]):  # the sides' mean over the seeds
            n, n2 = n + L ** 2, n2 + L ** 4
        return {"bytes": n * (8 + 64 + 16 + 16), "flops": n2 * 18 * 2 * (M // 2)}
    n, cols = case["lx"] * case["ly"], _columns(case)
    if kind in ("scf", "map", "slab"):
        return {"bytes": n * (8 + 64 + 16 + 24), "flops": case.get("iters", 1) * n * cols * 18 * 2 * (M // 2)}
    if kind == "ldos":
        return {"bytes": n * (8 + 64 + 16) + 4 * cols * case["energies"],
                "flops": n * cols * 18 * 2 * (M // 2) + 2 * cols * M * case["energies"]}
    if kind == "vortex_ldos":
        return {"bytes": n * (8 + 128 + 64) + 4 * cols * case["energies"],
                "flops": n * cols * 112 * 2 * M + 2 * cols * M * case["energies"]}
    if kind == "currents":
        return {"bytes": n * (8 + 128 + 64 + 64), "flops": n * cols * 112 * 2 * M}
    if kind == "green":
        pairs = cols * min(n, case["targets"])
        return {"bytes": n * (8 + 128 + 64) + 2 * 16 * pairs * case["energies"],
                "flops": n * cols * 112 * 2 * M + 2 * 8 * pairs * M * case["energies"]}
    # gradient: the recursion, its reverse and 12 sums a site and step
    return {"bytes": n * (8 + 64 + 16 + 16) + n * (8 + 64 + 16), "flops": n * cols * (12 + 12 + 12) * 2 * M}


# -------------------------------------------- the same in 64 bits, plain torch

_DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _matrix(p, delta):
    """H of the lattice as (rows, cols, values), electron row 2s, hole row 2s+1,
    and the labels that gradients need: (kind, site, direction)."""
    nd = p.hop.shape[1]
    nb = _neighbours(p.Lx, p.Ly, p.periodic_x, p.periodic_y, nd)
    s = np.arange(p.Lx * p.Ly)
    xi = p.eps - p.mu
    r, c, v, lab = [2 * s, 2 * s + 1], [2 * s, 2 * s + 1], [xi, -xi], [("ee", -1), ("hh", -1)]
    if p.pairing == 0:
        r += [2 * s, 2 * s + 1]
        c += [2 * s + 1, 2 * s]
        v += [delta, np.conj(delta)]
        lab += [("eh", -1), ("he", -1)]
    for d in range(nd):
        on = nb[:, d] >= 0
        i, j, t = s[on], nb[on, d], p.hop[on, d]
        r += [2 * i, 2 * i + 1]
        c += [2 * j, 2 * j + 1]
        v += [-t, np.conj(t)]
        lab += [("ee", d), ("hh", d)]
        if p.pairing == 1 and d < 4:
            z = delta.reshape(-1, 4)[on, d]
            r += [2 * i, 2 * i + 1]
            c += [2 * j + 1, 2 * j]
            v += [z, np.conj(z)]
            lab += [("eh", d), ("he", d)]
    parts = [len(x) for x in r]
    return np.concatenate(r), np.concatenate(c), np.concatenate([np.asarray(x, dtype=np.complex128) for x in v]), lab, parts


def _scaled(p, delta):
    """(H / a as CSR on the device, a): a = 1.1 x the largest row sum of |H|."""
    r, c, v, _, _ = _matrix(p, delta)
    n2 = 2 * p.Lx * p.Ly
    a = 1.1 * np.bincount(r, weights=np.abs(v), minlength=n2).max()
    real = not np.any(v.imag)
    v = torch.from_numpy((v.real if real else v) / a)
    h = torch.sparse_coo_tensor(torch.from_numpy(np.stack([r, c])), v, (n2, n2)).to(_DEV).coalesce().to_sparse_csr()
    return h, a


def _jackson(M):
    n = np.arange(M)
    q = math.pi / (M + 1)
    return ((M - n + 1) * np.cos(q * n) + np.sin(q * n) / math.tan(q)) / (M + 1)


def _coefficients(M, a, T, K):
    """Jackson-damped Chebyshev coefficients of tanh(a x / 2T), K nodes."""
    th = torch.arange(K, dtype=torch.float64, device=_DEV).add_(0.5).mul_(math.pi / K)
    f = torch.tanh(a * torch.cos(th) / (2.0 * T))
    cn = torch.stack([(f * torch.cos(n * th)).sum() / K for n in range(M)]).cpu().numpy()
    cn[1:] *= 2.0
    return _jackson(M) * cn


def _start(h, sites):
    j0 = torch.zeros((h.shape[0], len(sites)), dtype=h.dtype, device=_DEV)
    j0[2 * torch.as_tensor(np.asarray(sites), dtype=torch.int64, device=_DEV), torch.arange(len(sites), device=_DEV)] = 1.0
    return j0


def _vectors(h, sites, M):
    """j_0 .. j_{M-1}, one after the other."""
    a, b = _start(h, sites), None
    yield a
    b = torch.sparse.mm(h, a)
    yield b
    for _ in range(2, M):
        a = torch.sparse.mm(h, b).mul_(2.0).sub_(a)
        a, b = b, a
        yield b


def _chunks(n, per):
    return [np.arange(k, min(n, k + per)) for k in range(0, n, per)]


def _map_exact(p, delta, M, T, K, sites=None, U=None):
    """Delta_out and n at the start sites (all of them, on-site pairing)."""
    h, a = _scaled(p, delta)
    sites = np.arange(p.Lx * p.Ly) if sites is None else sites
    C = _coefficients(M, a, T, K)
    out_d = np.zeros(sites.size, dtype=np.complex128)
    out_n = np.ones(sites.size)
    for part in _chunks(sites.size, max(1, int(2.5e10 / (h.shape[0] * 16)))):
        at = torch.as_tensor(2 * sites[part], dtype=torch.int64, device=_DEV)
        col = torch.arange(part.size, device=_DEV)
        sd = torch.zeros(part.size, dtype=h.dtype, device=_DEV)
        sn = torch.zeros(part.size, dtype=h.dtype, device=_DEV)
        for m, j in enumerate(_vectors(h, sites[part], M)):
            sn += C[m] * j[at, col]
            sd += C[m] * j[at + 1, col].conj()
        out_d[part] = sd.cpu().numpy()
        out_n[part] -= sn.real.cpu().numpy()
    return 0.5 * (p.coupling if U is None else U) * out_d, out_n


def _moments_exact(p, sites, M):
    h, a = _scaled(p, p.delta0)
    at = torch.as_tensor(2 * sites.astype(np.int64), device=_DEV)
    col = torch.arange(sites.size, device=_DEV)
    return torch.stack([j[at, col].real for j in _vectors(h, sites, M)], 1).cpu().numpy(), a


def _ldos_exact(p, M, g):
    mu, a = _moments_exact(p, p.sites, M)
    x = p.energies / a
    w = g[:, None] * np.cos(np.arange(M)[:, None] * np.arccos(x))
    w[1:] *= 2.0
    return mu @ w / (math.pi * a * np.sqrt(1.0 - x * x))


def _grad_exact(p, M, T, K):
    """Gradients of sum Re(conj(weight) Delta_out) for on-site pairing."""
    h, a = _scaled(p, p.delta0)
    n, nd = p.Lx * p.Ly, p.hop.shape[1]
    C = _coefficients(M, a, T, K)
    r, c, _, lab, parts = _matrix(p, p.delta0)
    r, c = torch.from_numpy(r).to(_DEV), torch.from_numpy(c).to(_DEV)
    G = torch.zeros(r.numel(), dtype=h.dtype, device=_DEV)
    for part in _chunks(n, max(1, int(3e10 / (M * 2 * n * 16)))):
        j = list(_vectors(h, part, M))
        at = torch.as_tensor(2 * part + 1, dtype=torch.int64, device=_DEV)
        col = torch.arange(part.size, device=_DEV)
        y = torch.from_numpy(0.5 * p.coupling * np.conj(p.weight[part])).to(_DEV)
        y = y if h.is_complex() else y.real.contiguous()
        l1 = torch.zeros_like(j[0])
        l2 = torch.zeros_like(j[0])
        for m in range(M - 1, 0, -1):
            l1, l2 = torch.sparse.mm(h, l1).mul_(2.0).sub_(l2), l1
            l1[at, col] += C[m] * y
            for q in _chunks(r.numel(), 65536):
                G[q[0]:q[-1] + 1] += (1.0 if m == 1 else 2.0) * (
                    l1[r[q[0]:q[-1] + 1]] * j[m - 1][c[q[0]:q[-1] + 1]].conj()).sum(1)
    G = G.cpu().numpy() / a
    nb = _neighbours(p.Lx, p.Ly, p.periodic_x, p.periodic_y, nd)
    g = {k: np.zeros((n, nd), dtype=np.complex128) for k in ("ee", "hh")}
    eps, delta, k0 = np.zeros(n), np.zeros(n, dtype=np.complex128), 0
    for (what, d), cnt in zip(lab, parts):
        part, k0 = G[k0:k0 + cnt], k0 + cnt
        if d >= 0:
            g[what][nb[:, d] >= 0, d] = part
        elif what in ("ee", "hh"):
            eps += part.real if what == "ee" else -part.real
        else:
            delta += part if what == "eh" else np.conj(part)
    hop = np.zeros((n, nd), dtype=np.complex128)
    for d in range(nd):
        on = nb[:, d] >= 0
        j = nb[on, d]
        hop[on, d] = (-g["ee"][on, d] - np.conj(g["ee"][j, d ^ 1]) + np.conj(g["hh"][on, d]) + g["hh"][j, d ^ 1])
    return {"eps": eps, "hop": hop, "delta": delta}


def _seconds(case):
    """What exact() would take: two passes over the vectors a moment at about
    2 TB/s (sparse products), some more for the gradient's sums."""
    if case["kind"] == "ensemble":
        pairs = sum(L ** 4 for L in np.linspace(case["lo"], case["hi"], case["members"]))
        return pairs * 2 * 8 * case["M"] * 4 / 2e12
    pairs = case["lx"] * case["ly"] * _columns(case)
    wide = 2 if case["kind"] in ("vortex_ldos", "currents", "green") else 1
    return pairs * 2 * 8 * wide * case["M"] * case.get("iters", 1) * (30 if case["kind"] == "grad" else 6) / 2e12


def exact(case, seed):
    if _seconds(case) > 20.0:
        return None
    p, kind, M = _problem(case, seed), case["kind"], case["M"]
    if kind == "ensemble":
        return [q.delta0 + 0.5 * (_map_exact(q, q.delta0, M, q.T, 16384)[0] - q.delta0) for q in p]
    if kind == "scf":
        delta, moved = p.delta0.copy(), []
        for _ in range(case["iters"]):
            out = _map_exact(p, delta, M, p.T, 65536)[0]
            moved.append(np.abs(out - delta).max())
            delta = delta + 0.5 * (out - delta)
        return {"delta": delta, "moved": np.array(moved)}
    if kind == "map":
        delta, n = _map_exact(p, p.delta0, M, p.T, 65536)
        return {"delta": delta, "n": n}
    if kind == "slab":
        reps = np.arange(p.Ly) * p.Lx
        delta, n = _map_exact(p, p.delta0, M, p.T, 65536, sites=reps, U=p.U_site[reps])
        return {"delta": np.repeat(delta, p.Lx), "n": np.repeat(n, p.Lx)}
    if kind == "ldos":
        _, a = _scaled(p, p.delta0)
        lam = 0.01 * M / a
        k = 1.0 - np.arange(M) / M
        return _ldos_exact(p, M, np.sinh(lam * k) / math.sinh(lam))
    if kind == "vortex_ldos":
        return _ldos_exact(p, M, _jackson(M))
    if kind == "grad":
        return _grad_exact(p, M, p.T, 65536)
    h, a = _scaled(p, p.delta0)
    if kind == "currents":
        C = _coefficients(M, a, p.T, 65536)
        nb = torch.from_numpy(_neighbours(p.Lx, p.Ly, 1, 1, p.hop.shape[1])).to(_DEV)
        n = p.Lx * p.Ly
        acc = torch.zeros((n, p.hop.shape[1]), dtype=h.dtype, device=_DEV)
        for part in _chunks(n, max(1, int(2.5e10 / (2 * n * 16)))):
            col = torch.arange(part.size, device=_DEV)[:, None]
            for m, j in enumerate(_vectors(h, part, M)):
                acc[part[0]:part[-1] + 1] += C[m] * j[2 * nb[part[0]:part[-1] + 1], col]
        return -2.0 * (p.hop * acc.cpu().numpy()).imag
    # nonlocal Green's functions
    at = torch.as_tensor(2 * p.targets.astype(np.int64), device=_DEV)
    e, q = [], []
    for j in _vectors(h, p.sites, M):
        e.append(j[at].T.clone())
        q.append(j[at + 1].T.clone())
    x = p.energies / a
    th = np.arccos(x)
    w = _jackson(M)[:, None] * np.exp(-1j * np.arange(M)[:, None] * th) * (-2j / (a * np.sqrt(1.0 - x * x)))
    w[0] *= 0.5
    w = torch.from_numpy(w).to(_DEV)
    return [torch.einsum("mst,me->ste", torch.stack(z).to(torch.complex128), w) for z in (e, q)]
