"""Performance cases of the sCOLA library: the calls its users make, over their real range of sizes.

A case names a kind of call ("kind") and a problem statement (the keyword arguments of
``Scola`` plus a few numbers of its own):

  forward   Scola.forward: a whole run from white noise; momenta and displacements
  gradient  ScolaState: a checkpointed run and the VJP of its final state with respect to the noise
  tcola     Scola.tcola: the periodic full-box run of the same particles
  force     Scola.pm_force: one particle-mesh force evaluation of every box (deposit, Dirichlet
            solve, gradient and interpolation), the inner layer of every run
  lpt       Scola.lpt_fields: the full-box initial conditions and 2LPT stage
  density   Scola.final_density and its adjoint: the analysis end of a differentiated pipeline

Final positions are compared as displacements x - q wrapped to the nearest image: a particle on a
face of the box may leave either call at 0 or at L.  Whole runs take particle spacings above
3 Mpc/h (large-volume mocks), where a change of the last bit of one force does not grow along a
collapsed orbit; the single force evaluations cover the denser boxes and the latest times.
"""
import functools
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import paper_2003_04925_gb300 as sc

COSMOLOGY = dict(Om=0.3, OL=0.7, h=0.7, ns=0.96, sigma8=0.8)
NLPT = -2.5


def listed():
    return [
        # a quick run on a laptop-sized box, 8 boxes of 24^3 particles and cells: launch-bound
        dict(name="forward_32", kind="forward", L=100.0, Np=32, Ntiles=2, Nbuf=4, mesh_ratio=1, nsteps=10, a_i=0.02,
             a_f=1.0),
        # a large-volume mock at z = 1, 64 boxes on 96^3 meshes (two cells per particle spacing): the main use
        dict(name="forward_128", kind="forward", L=1000.0, Np=128, Ntiles=4, Nbuf=8, mesh_ratio=2, nsteps=20, a_i=0.02,
             a_f=0.5),
        # one gradient of a field-level inference chain, 64 boxes on 48^3 meshes
        dict(name="gradient_128", kind="gradient", L=500.0, Np=128, Ntiles=4, Nbuf=8, mesh_ratio=1, nsteps=10,
             a_i=0.02, a_f=0.5),
        # the monolithic run that the tiles are compared with, on a 256^3 mesh
        dict(name="tcola_128", kind="tcola", L=1000.0, Np=128, Ntiles=4, Nbuf=8, mesh_ratio=2, nsteps=10, a_i=0.02,
             a_f=1.0),
        # initial conditions alone
        dict(name="lpt_128", kind="lpt", L=250.0, Np=128, Ntiles=4, Nbuf=8, mesh_ratio=1),
        # final density of a 256^3 run and the adjoint of a loss of it
        dict(name="density_256", kind="density", L=500.0, Np=256, Ntiles=4, Nbuf=4, mesh_ratio=1, a=1.0),
        # force evaluations, from the smallest call to the largest: 8 boxes of 24^3 cells
        dict(name="force_24", kind="force", L=100.0, Np=32, Ntiles=2, Nbuf=4, mesh_ratio=1, a=1.0),
        # fourth-order differences on 64 boxes of 48^3 cells
        dict(name="force_48_fda4", kind="force", L=250.0, Np=128, Ntiles=4, Nbuf=8, mesh_ratio=1, fda_order=4, a=0.5),
        # the dense late-time boxes of a 2 Mpc/h run, 64 boxes on 96^3 meshes
        dict(name="force_96", kind="force", L=250.0, Np=128, Ntiles=4, Nbuf=8, mesh_ratio=2, a=1.0),
        # a buffer width per tile: meshes of 72, 80 and 96 cells in the same launches
        dict(name="force_uneven", kind="force", L=500.0, Np=256, Ntiles=4, buffer_seed=7, mesh_ratio=1, a=1.0),
        # one mesh cell more than particles per side, as in the 1 Gpc/h runs: odd meshes of 189 cells
        dict(name="force_189", kind="force", L=250.0, Np=256, Ntiles=2, Nbuf=30, Ng=189, a=0.5),
        # the largest meshes of the production configuration, 192^3, on one of the shares of a sharded run
        dict(name="force_192", kind="force", L=250.0, Np=256, Ntiles=4, Nbuf=16, mesh_ratio=2, box_first=16,
             box_count=16, a=1.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _tiling(rng, max_particles, max_ng, cells_max, ratios=(1, 1, 2)):
    """A random tiling: particles per side, tiles, a buffer and a mesh within the given limits."""
    while True:
        nt = rng.choice((1, 2, 2, 3, 4, 4))
        ntile = int(round(_log(rng, 10, 96)))
        npart = nt * ntile
        nbuf = 0 if nt == 1 else int(round(_log(rng, 2, 32)))
        nsc = ntile + 2 * nbuf
        ratio = rng.choice(ratios)
        extra = rng.choice((0, 0, 1)) if ratio == 1 else 0
        ng = ratio * nsc + extra
        if nsc > npart or npart > max_particles or not 12 <= ng <= max_ng or nt**3 * ng**3 > cells_max:
            continue
        c = dict(Np=npart, Ntiles=nt, Nbuf=nbuf)
        c.update(dict(Ng=ng) if extra else dict(mesh_ratio=ratio))
        return c


def draw(rng):
    kind = rng.choice(("force",) * 5 + ("forward", "forward", "gradient", "tcola", "lpt", "density"))
    if kind == "force":
        if rng.random() < 0.25:            # a buffer width per tile
            ntile = rng.choice((16, 24, 32, 40, 48, 64))
            c = dict(Np=4 * ntile, Ntiles=4, buffer_seed=rng.randrange(1000), mesh_ratio=1)
        else:
            c = _tiling(rng, 256, 220, 1.1e8)
            c["fda_order"] = rng.choice((2, 2, 2, 2, 4, 6))
        c.update(kind=kind, L=round(c["Np"] * _log(rng, 0.9, 6.0), 3), a=round(rng.uniform(0.1, 1.0), 3))
        return c
    if kind in ("lpt", "density"):
        n = int(round(_log(rng, 24, 256)))
        c = dict(kind=kind, Np=n, Ntiles=1, Nbuf=0, mesh_ratio=1, L=round(n * _log(rng, 1.5, 8.0), 3))
        if kind == "density":
            c["a"] = round(rng.uniform(0.2, 1.0), 3)
        return c
    c = dict(kind=kind, a_i=0.02, a_f=round(rng.uniform(0.3, 0.6), 3), nsteps=rng.randint(8, 12))
    if kind == "tcola":
        ratio = rng.choice((1, 2))
        n = int(round(_log(rng, 24, 128)))
        c.update(Np=n, Ntiles=1, Nbuf=0, mesh_ratio=ratio)
    else:
        c.update(_tiling(rng, 128, 128, 3e7, (1, 1, 2) if kind == "forward" else (1,)))
    two = c.get("mesh_ratio", 1) == 2
    c["L"] = round(c["Np"] * (_log(rng, 7.0, 10.0) if two else _log(rng, 3.0, 8.0)), 3)
    return c


# ---------------------------------------------------------------- geometry and inputs

def _buffers(c):
    n = c["Ntiles"] ** 3
    if "buffer_seed" in c:
        r = np.random.RandomState(c["buffer_seed"])
        return [int(b) for b in r.choice((4, 8, 16), size=n)]
    return [c["Nbuf"]] * n


def _boxes(c):
    """(tile coordinates, buffer, particles per side, cells per side) of every box of the context."""
    t, nt = c["Ntiles"], c["Np"] // c["Ntiles"]
    out = []
    for b, buf in enumerate(_buffers(c)):
        nsc = nt + 2 * buf
        out.append(((b // (t * t), b // t % t, b % t), buf, nsc, c["Ng"] if c.get("Ng") else c["mesh_ratio"] * nsc))
    f = c.get("box_first", 0)
    return out[f:f + c["box_count"]] if c.get("box_count") else out


def _params(c):
    kw = dict(COSMOLOGY)
    for k in ("L", "Np", "Ntiles", "Nbuf", "mesh_ratio", "Ng", "fda_order", "nsteps", "a_i", "a_f", "box_first",
              "box_count"):
        if k in c:
            kw[k] = c[k]
    kw.setdefault("nsteps", 1)
    kw.setdefault("a_i", 0.02)
    kw.setdefault("a_f", 1.0)
    if "buffer_seed" in c:
        kw.update(Nbuf=0, buffers=_buffers(c))
    return kw


def _noise(c, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    n = c["Np"]
    return torch.randn(n, n, n, generator=g, device="cuda", dtype=torch.float32)


def _ids(c, box):
    """Global ids of a box's particles, box-local order."""
    t, buf, nsc, _ = box
    n, nt = c["Np"], c["Np"] // c["Ntiles"]
    r = torch.arange(nsc, device="cuda")
    x, y, z = ((ta * nt - buf + r) % n for ta in t)
    return ((x[:, None, None] * n + y[None, :, None]) * n + z[None, None, :]).reshape(-1)


def _lattice(n, d):
    r = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * d
    return torch.stack(torch.meshgrid(r, r, r, indexing="ij")).reshape(3, -1)


def _displacements(c, seed):
    """2LPT displacements (3, Np^3) at scale factor c["a"], in 64 bits from another field than the shells'."""
    _, _, _, psi1, psi2 = _lpt64(c, _noise(c, seed + 500_000))
    g = _growth([c["a"]])
    return -g["D1"][0] * psi1 + g["D2"][0] * psi2


def _box_displacements(c, seed):
    """The displacements of every box particle, (3, P) FP32, boxes concatenated."""
    s = _displacements(c, seed)
    return torch.cat([s[:, _ids(c, b)].float() for b in _boxes(c)], 1).contiguous()


def _cotangents(c, seed):
    """Smooth cotangents of final positions and momenta, (Np^3, 3) each: those of large-scale modes."""
    r = np.random.RandomState(seed % (1 << 31))
    q = _lattice(c["Np"], 1.0 / c["Np"])
    out = []
    for _ in range(2):
        v = torch.zeros_like(q)
        for _ in range(4):
            k = torch.tensor(r.randint(-3, 4, size=3), device="cuda", dtype=torch.float64)
            amp = torch.tensor(r.standard_normal(3), device="cuda", dtype=torch.float64)
            v += amp[:, None] * torch.sin(2 * math.pi * (k @ q) + r.uniform(0, 2 * math.pi))
        out.append(v.T.float().contiguous())
    return out


def _periodic_positions(c, seed):
    """Final positions of a run at c["a"], (Np^3, 3) FP32 in [0, L)."""
    x = (_lattice(c["Np"], c["L"] / c["Np"]) + _displacements(c, seed)).T.float().remainder(c["L"])
    return torch.where(x < c["L"], x, torch.zeros_like(x)).contiguous()


def prepare(case, seed):
    c, kind = dict(case), case["kind"]
    sim = sc.Scola(**_params(c))
    st = dict(kind=kind, sim=sim, L=c["L"])
    if kind == "density":
        st["x"] = _periodic_positions(c, seed)
        st["lam"] = _noise(c, seed + 1)
        return st
    st["w"] = _noise(c, seed)
    if kind in ("forward", "tcola"):
        st["q"] = _lattice(c["Np"], c["L"] / c["Np"]).T.float().contiguous()
    if kind == "gradient":
        st["w"].requires_grad_(True)
        st["gx"], st["gp"] = _cotangents(c, seed)
    if kind == "force":
        st["s"] = _box_displacements(c, seed)
        st["D1"] = _growth([c["a"]])["D1"][0]
        sim.lpt_fields(st["w"])
        sim.setup_boxes()
    return st


def run(state):
    kind, sim = state["kind"], state["sim"]
    if kind in ("forward", "tcola"):
        x, p = (sim.forward if kind == "forward" else sim.tcola)(state["w"])
        d = x.sub_(state["q"])
        d.sub_(torch.round(d / state["L"]), alpha=state["L"])
        return {"p": p, "displacement": d}
    if kind == "gradient":
        x, p = sc.ScolaState.apply(state["w"], sim)
        (g,) = torch.autograd.grad((x, p), (state["w"],), (state["gx"], state["gp"]))
        return {"p": p.detach(), "gradient": g}
    if kind == "force":
        return {"F": sim.pm_force(state["s"], state["D1"])[0]}
    if kind == "lpt":
        return sim.lpt_fields(state["w"])
    return {"delta": sim.final_density(state["x"]), "lam_x": sim.density_adjoint(state["x"], state["lam"])}


def work(case):
    """Bytes and operations of one pass.  A run streams its box particles (84 bytes each: state read and
    written, frame and positions read) and its meshes (source and potential, written and read once) at
    every force evaluation, since neither stays on chip; a transform of a pencil takes 2.5 n log2 n."""
    c, kind = case, case["kind"]
    n3 = c["Np"] ** 3
    fft = 2.5 * n3 * math.log2(n3)
    if kind == "density":
        return {"bytes": 12 * n3 + 4 * n3 + 12 * n3 + 4 * n3 + 12 * n3, "flops": 100 * n3}
    if kind == "lpt":
        return {"bytes": 4 * n3 + 9 * 4 * n3, "flops": 10 * fft + 60 * n3}
    if kind == "tcola":
        m = (c["mesh_ratio"] * c["Np"]) ** 3
        per = {"bytes": 84 * n3 + 16 * m, "flops": 200 * n3 + 5 * m * math.log2(m)}
    else:
        boxes = _boxes(c)
        P = sum(b[2] ** 3 for b in boxes)
        M = sum(b[3] ** 3 for b in boxes)
        solve = sum(6 * 2.5 * b[3] ** 3 * math.log2(b[3] + 1) for b in boxes)
        if kind == "force":
            return {"bytes": 24 * P + 16 * M, "flops": 200 * P + solve}
        per = {"bytes": 84 * P + 16 * M, "flops": 200 * P + solve}
    k = (c["nsteps"] + 1) * (3 if kind == "gradient" else 1)
    return {"bytes": 28 * n3 + k * per["bytes"], "flops": 12 * fft + k * per["flops"]}


# ---------------------------------------------------------------- the same results in 64 bits

_G = {2: (1 / 2,), 4: (2 / 3, -1 / 12), 6: (3 / 4, -3 / 20, 1 / 60)}
_S = {2: (-2, 1), 4: (-5 / 2, 4 / 3, -1 / 12), 6: (-49 / 18, 3 / 2, -3 / 20, 1 / 90)}


def _hubble(a):
    Om, OL = COSMOLOGY["Om"], COSMOLOGY["OL"]
    return np.sqrt(Om / a + (1 - Om - OL) + OL * a * a)


def _growth(a):
    return _growth_at(tuple(float(v) for v in a))


@functools.lru_cache(maxsize=64)
def _growth_at(a, steps=3000, a0=1e-6):
    """D1, D2 and their derivatives dD/da at the scale factors a, D1(1) = 1 (RK4 in ln a)."""
    Om, OL = COSMOLOGY["Om"], COSMOLOGY["OL"]
    t = np.concatenate([np.asarray(a, np.float64), [1.0]])

    def rhs(y, S):
        x = np.exp(y)
        E2 = Om / x**3 + (1 - Om - OL) / x**2 + OL
        f = 2 + (-3 * Om / x**3 - 2 * (1 - Om - OL) / x**2) / (2 * E2)
        g = 1.5 * Om / x**3 / E2
        return np.array([S[1], -f * S[1] + g * S[0], S[3], -f * S[3] + g * (S[2] - S[0] ** 2)])

    y = np.full_like(t, math.log(a0))
    h = (np.log(t) - y) / steps
    one = np.ones_like(t)
    S = np.array([a0 * one, a0 * one, -3 / 7 * a0**2 * one, -6 / 7 * a0**2 * one])
    for _ in range(steps):
        k1 = rhs(y, S)
        k2 = rhs(y + h / 2, S + h / 2 * k1)
        k3 = rhs(y + h / 2, S + h / 2 * k2)
        k4 = rhs(y + h, S + h * k3)
        S, y = S + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4), y + h
    n = S[0, -1]
    return {"D1": (S[0] / n)[:-1], "D2": (S[2] / n**2)[:-1], "d1": (S[1] / n / t)[:-1], "d2": (S[3] / n**2 / t)[:-1]}


def _schedule(c):
    """Time factors of the kick-drift-kick sequence, steps linear in a, u(a) = a^nLPT."""
    n, ai, af, Om = c["nsteps"], c["a_i"], c["a_f"], COSMOLOGY["Om"]
    a = ai + (af - ai) * np.arange(n + 1) / n
    ah = (a[1:] + a[:-1]) / 2
    lo, hi = np.concatenate([a[:1], ah]), np.concatenate([ah, a[-1:]])
    g = dict(_growth(a))
    x, wq = np.polynomial.legendre.leggauss(48)
    alpha = []
    for k in range(n):
        z = (a[k + 1] - a[k]) / 2 * x + ah[k]
        alpha.append(ah[k] ** -NLPT * (a[k + 1] - a[k]) / 2 * np.sum(wq * z ** (NLPT - 2) / _hubble(z)))
    g.update(a=a, alpha=alpha, beta=-1.5 * Om * (hi**NLPT - lo**NLPT) / (NLPT * a**NLPT * _hubble(a)))
    return g


@functools.lru_cache(maxsize=1)
def _amplitude():
    """A of P = A k^ns T^2 from sigma8 (Simpson's rule in ln k)."""
    m = 1 << 20
    lk = np.linspace(math.log(1e-5), math.log(1e3), m + 1)
    k = np.exp(lk)
    x = 8 * k
    W = np.where(x > 1e-2, 3 * (np.sin(x) - x * np.cos(x)) / x**3, 1 - x * x / 10 + x**4 / 280)
    f = k**3 * _unnormalised(torch.from_numpy(k)).numpy() * W**2 / (2 * math.pi**2)
    integral = (lk[1] - lk[0]) / 3 * (f[0] + f[-1] + 4 * f[1:-1:2].sum() + 2 * f[2:-1:2].sum())
    return COSMOLOGY["sigma8"] ** 2 / integral


def _unnormalised(k):
    q = k / (COSMOLOGY["Om"] * COSMOLOGY["h"])
    T = torch.log1p(2.34 * q) / (2.34 * q) * (1 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3
                                              + (6.71 * q) ** 4) ** -0.25
    return k ** COSMOLOGY["ns"] * T * T


def _gradient64(phi, d, order):
    return torch.stack([sum(g * (phi.roll(-m, ax) - phi.roll(m, ax)) for m, g in enumerate(_G[order], 1)) / d
                        for ax in range(3)])


def _lpt64(c, w):
    """delta, phi1, phi2 (N^3 each), psi1 and psi2 (3, N^3 flattened) of the white noise w."""
    N, order = c["Np"], c.get("fda_order", 2)
    d = c["L"] / N
    w = w.double()
    f = torch.fft.fftfreq(N, 1 / N, device="cuda", dtype=torch.float64)
    fz = torch.fft.rfftfreq(N, 1 / N, device="cuda", dtype=torch.float64)
    ax = (f[:, None, None], f[None, :, None], fz[None, None, :])
    k = 2 * math.pi / c["L"] * torch.sqrt(sum(v * v for v in ax))
    k[0, 0, 0] = 1.0
    amp = torch.sqrt(_amplitude() * _unnormalised(k) / d**3)
    amp[0, 0, 0] = 0.0
    kd = [2 * math.pi / N * v for v in ax]
    lam = sum(2 * sum(s * (torch.cos(m * v) - 1) for m, s in enumerate(_S[order]) if m) / d**2 for v in kd)
    lam[0, 0, 0] = 1.0
    inv = 1 / lam
    inv[0, 0, 0] = 0.0
    D = [2 / d * sum(g * torch.sin(m * v) for m, g in enumerate(_G[order], 1)) for v in kd]
    dk = torch.fft.rfftn(w) * amp
    pk = dk * inv

    def back(x):
        return torch.fft.irfftn(x, s=(N, N, N))

    def second(i, j):
        return back(-D[i] * D[j] * pk)

    phi1 = back(pk)
    xx, yy, zz = second(0, 0), second(1, 1), second(2, 2)
    src = xx * yy + xx * zz + yy * zz - second(0, 1) ** 2 - second(0, 2) ** 2 - second(1, 2) ** 2
    phi2 = back(torch.fft.rfftn(src) * inv)
    return back(dk), phi1, phi2, _gradient64(phi1, d, order).reshape(3, -1), _gradient64(phi2, d, order).reshape(3, -1)


def _corners(u, top=None):
    """(lower corner, weights of the 8 corners with their offsets) of mesh coordinates u (3, n)."""
    i0 = torch.floor(u.detach())
    if top is not None:
        i0 = torch.clamp(i0, max=float(top))
    f = u - i0
    out = []
    for o in range(8):
        e = (o >> 2, o >> 1 & 1, o & 1)
        out.append((e, math.prod((f[a] if e[a] else 1 - f[a]) for a in range(3))))
    return i0.long(), out


def _shell64(c, box, phi1):
    """phi1 interpolated to the padded cells of a box, zero inside."""
    t, buf, nsc, ng = box
    n, nt, P = c["Np"], c["Np"] // c["Ntiles"], c.get("fda_order", 2)
    cell = torch.arange(-P, ng + P, device="cuda", dtype=torch.float64)
    idx, wt = [], []
    for ta in t:
        u = (ta * nt - buf) + (cell + 0.5) * nsc / ng - 0.5
        i = torch.floor(u)
        idx.append((i.long() % n, (i.long() + 1) % n))
        wt.append((1 - (u - i), u - i))
    out = 0
    for o in range(8):
        e = (o >> 2, o >> 1 & 1, o & 1)
        w = [wt[a][e[a]] for a in range(3)]
        out = out + (w[0][:, None, None] * w[1][None, :, None] * w[2][None, None, :]
                     * phi1[idx[0][e[0]][:, None, None], idx[1][e[1]][None, :, None], idx[2][e[2]][None, None, :]])
    mask = torch.ones_like(out)
    mask[P:-P, P:-P, P:-P] = 0
    return out * mask


def _force64(c, nsc, ng, s, shell, D1):
    """grad Phi (3, n) at a box's particles with displacements s (3, n)."""
    P = c.get("fda_order", 2)
    dq = c["L"] / c["Np"]
    dg = nsc * dq / ng
    x = (_lattice(nsc, dq) + s) / dg - 0.5
    i0, corners = _corners(x)
    rho = torch.zeros(ng**3, dtype=torch.float64, device="cuda")
    for e, w in corners:
        cell = [i0[a] + e[a] for a in range(3)]
        ok = sum(((v >= 0) & (v < ng)).long() for v in cell) == 3
        flat = torch.where(ok, (cell[0] * ng + cell[1]) * ng + cell[2], torch.zeros_like(cell[0]))
        rho = rho.index_add(0, flat, torch.where(ok, w, torch.zeros_like(w)))
    src = rho.reshape(ng, ng, ng) * (ng / nsc) ** 3 - 1
    bc = D1 * shell
    inner = slice(P, ng + P)
    for m, sm in enumerate(_S[P]):
        if m:
            lo, hi = slice(P - m, ng + P - m), slice(P + m, ng + P + m)
            src = src - sm / dg**2 * (bc[lo, inner, inner] + bc[hi, inner, inner] + bc[inner, lo, inner]
                                      + bc[inner, hi, inner] + bc[inner, inner, lo] + bc[inner, inner, hi])
    i = torch.arange(1, ng + 1, device="cuda", dtype=torch.float64)
    S = torch.sin(math.pi / (ng + 1) * (i[:, None] * i[None, :] % (2 * ng + 2)))
    lam = 2 / dg**2 * sum(sm * (torch.cos(math.pi * m * i / (ng + 1)) - 1) for m, sm in enumerate(_S[P]) if m)

    def dst(v):
        v = torch.matmul(torch.matmul(S, v), S)
        return torch.matmul(S, v.reshape(ng, -1)).reshape(ng, ng, ng)

    phi = dst(dst(src) / (lam[:, None, None] + lam[None, :, None] + lam[None, None, :])) * (8 / (ng + 1) ** 3)
    phi = (bc + torch.nn.functional.pad(phi, (P,) * 6)).reshape(-1)
    nh, side = P // 2, ng + 2 * P
    u = torch.clamp(x, -float(nh), float(ng + nh - 1))
    i0, corners = _corners(u, ng + nh - 2)
    F = [0.0, 0.0, 0.0]
    for e, w in corners:
        at = ((i0[0] + e[0] + P) * side + (i0[1] + e[1] + P)) * side + i0[2] + e[2] + P
        for a, st in enumerate((side * side, side, 1)):
            for m, g in enumerate(_G[P], 1):
                F[a] = F[a] + w * (g / dg) * (phi[at + m * st] - phi[at - m * st])
    return torch.stack(F)


def _kdk64(c, s, psi1, psi2, sched, force):
    """The kick-drift-kick sequence; final displacements and momenta (frame added back)."""
    p = torch.zeros_like(s)

    def step(k, s, p):
        D1, D2 = sched["D1"][k], sched["D2"][k]
        p = p + sched["beta"][k] * (force(s, D1) - D1 * psi1 + (D2 - D1 * D1) * psi2)
        if k < c["nsteps"]:
            s = (s + sched["alpha"][k] * p - (sched["D1"][k + 1] - D1) * psi1 + (sched["D2"][k + 1] - D2) * psi2)
        return s, p

    for k in range(c["nsteps"] + 1):
        s, p = checkpoint(step, k, s, p, use_reentrant=False) if s.requires_grad else step(k, s, p)
    af = c["a_f"]
    return s, p + af * af * _hubble(af) * (-sched["d1"][-1] * psi1 + sched["d2"][-1] * psi2)


def _run64(c, w):
    """Final displacements and momenta (3, Np^3) of a tiled run."""
    _, phi1, _, psi1, psi2 = _lpt64(c, w)
    sched = _schedule(c)
    s_out, p_out, order = [], [], []
    for box in _boxes(c):
        t, buf, nsc, ng = box
        ids = _ids(c, box)
        q1, q2 = psi1[:, ids], psi2[:, ids]
        shell = _shell64(c, box, phi1)
        s, p = _kdk64(c, -sched["D1"][0] * q1 + sched["D2"][0] * q2, q1, q2, sched,
                      lambda s, D1, nsc=nsc, ng=ng, shell=shell: _force64(c, nsc, ng, s, shell, D1))
        keep = torch.zeros(nsc, nsc, nsc, dtype=torch.bool, device="cuda")
        keep[buf:nsc - buf, buf:nsc - buf, buf:nsc - buf] = True
        keep = keep.reshape(-1)
        s_out.append(s[:, keep])
        p_out.append(p[:, keep])
        order.append(ids[keep])
    back = torch.argsort(torch.cat(order))
    return torch.cat(s_out, 1)[:, back], torch.cat(p_out, 1)[:, back]


def _periodic_density(x, n, npart):
    """Periodic CIC density contrast on n^3 cells of mesh coordinates x (3, m)."""
    i0, corners = _corners(x)
    rho = torch.zeros(n**3, dtype=torch.float64, device="cuda")
    for e, w in corners:
        cell = [(i0[a] + e[a]) % n for a in range(3)]
        rho = rho.index_add(0, (cell[0] * n + cell[1]) * n + cell[2], w)
    return rho.reshape(n, n, n) * (n / npart) ** 3 - 1


def _tcola64(c, w):
    _, _, _, psi1, psi2 = _lpt64(c, w)
    sched = _schedule(c)
    n = c["mesh_ratio"] * c["Np"]
    dg = c["L"] / n
    q = _lattice(c["Np"], c["L"] / c["Np"])
    f = 2 * math.pi / n * torch.fft.fftfreq(n, 1 / n, device="cuda", dtype=torch.float64)
    fz = 2 * math.pi / n * torch.fft.rfftfreq(n, 1 / n, device="cuda", dtype=torch.float64)
    lam = 2 / dg**2 * ((torch.cos(f) - 1)[:, None, None] + (torch.cos(f) - 1)[None, :, None]
                       + (torch.cos(fz) - 1)[None, None, :])
    lam[0, 0, 0] = 1.0
    inv = 1 / lam
    inv[0, 0, 0] = 0.0

    def force(s, D1):
        u = (q + s) / dg - 0.5
        phi = torch.fft.irfftn(torch.fft.rfftn(_periodic_density(u, n, c["Np"])) * inv, s=(n, n, n))
        grad = _gradient64(phi, dg, 2).reshape(3, -1)
        i0, corners = _corners(u)
        F = 0
        for e, w in corners:
            cell = [(i0[a] + e[a]) % n for a in range(3)]
            F = F + w * grad[:, (cell[0] * n + cell[1]) * n + cell[2]]
        return F

    return _kdk64(c, -sched["D1"][0] * psi1 + sched["D2"][0] * psi2, psi1, psi2, sched, force)


def exact(case, seed):
    c, kind = dict(case), case["kind"]
    if kind == "density":
        x = _periodic_positions(c, seed).double().requires_grad_(True)
        delta = _periodic_density(x.T / (c["L"] / c["Np"]) - 0.5, c["Np"], c["Np"])
        (lam,) = torch.autograd.grad(delta, x, _noise(c, seed + 1).double())
        return {"delta": delta.detach(), "lam_x": lam}
    w = _noise(c, seed)
    if kind == "lpt":
        delta, phi1, phi2, psi1, psi2 = _lpt64(c, w)
        shape = (3,) + (c["Np"],) * 3
        return {"delta": delta, "phi1": phi1, "phi2": phi2, "psi1": psi1.reshape(shape), "psi2": psi2.reshape(shape)}
    if kind == "force":
        s, D1 = _box_displacements(c, seed), _growth([c["a"]])["D1"][0]
        phi1 = _lpt64(c, w)[1]
        out, at = [], 0
        for box in _boxes(c):
            n = box[2] ** 3
            out.append(_force64(c, box[2], box[3], s[:, at:at + n].double(), _shell64(c, box, phi1), D1))
            at += n
        return {"F": torch.cat(out, 1)}
    if kind == "gradient":
        w = w.double().requires_grad_(True)
        gx, gp = _cotangents(c, seed)
        s, p = _run64(c, w)
        (g,) = torch.autograd.grad((s, p), (w,), (gx.T.double(), gp.T.double()))
        return {"p": p.T.detach(), "gradient": g}
    s, p = (_run64 if kind == "forward" else _tcola64)(c, w)
    return {"p": p.T, "displacement": s.T}
