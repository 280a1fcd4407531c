"""Performance cases: the spectral requests a user of the library makes, through its C ABI binding.

Each case is one request (or one batch of served requests) on a lattice handle that the program
keeps: sizes from the repository's own workloads (64 x 64 square, 2048 x 2048 graphene with 4096
moments, vacancy graphene with time blocks and 64 energies, the dense D_H = 235 sample, disordered
graphene with optical conductivity, the serving stream of mixed lattices), shortened in the number
of moments or time steps where the full request would take seconds: the work per step is the same.

Outputs are kept in the precision that the request asks for: a complex64 request's numbers are
single precision whatever the width of the host buffer they arrive in, a complex128 request's are
double.  exact() evaluates the definitions in 64 bits with torch alone (its own Philox draws,
neighbour tables, Chebyshev series and current operator).
"""
from __future__ import annotations

import math
import random
import weakref

import numpy as np
import torch

from paper_2510_17432_gb300 import capi

SQUARE, HONEYCOMB, CUBIC = capi.SQUARE, capi.HONEYCOMB, capi.CUBIC
COORD = {SQUARE: 4, HONEYCOMB: 3, CUBIC: 6}
DENSE_DECAY = 0.3187  # 0.184 lattice constants of graphene, the decay of the pz model
DENSE_CUTOFF = {61: 5.1, 124: 7.1, 235: 9.7}
SQ3 = math.sqrt(3.0)

BASE = {"call": "dos", "kind": HONEYCOMB, "Lx": 1, "Ly": 1, "Lz": 1, "px": True, "py": True, "pz": True, "t": 1.0,
        "W": 0.0, "vac": 0.0, "dh": 0, "c128": False, "S": 1, "sites": False, "M": 0, "Nt": 0, "nE": 0,
        "method": "jackson", "tensor": False, "kT": 0.0, "mix": 0}


def _case(name=None, **kw):
    c = dict(BASE, **kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest configuration: one state on a 64 x 64 lattice in complex128, DOS (latency, launches)
        _case("square64_c128_dos", kind=SQUARE, Lx=64, Ly=64, W=1.0, c128=True, S=1, M=1024, nE=1024),
        # the small end of a request stream: an open ribbon of a few thousand sites, odd sizes
        _case("ribbon45x47_dos", Lx=45, Ly=47, py=False, W=1.0, S=4, M=512, nE=1024),
        # the headline workload: clean graphene, 8 states, 4096 moments, tensor-core reconstruction
        _case("graphene2048_dos", Lx=2048, Ly=2048, t=-2.7, S=8, M=4096, nE=8192, tensor=True),
        # a very large disordered sample (134M sites), as many moments as a second allows
        _case("graphene8192_dos", Lx=8192, Ly=8192, t=-2.7, W=1.0, S=4, M=256, nE=2048),
        # a disordered square lattice of odd size, a number of states that is no power of two
        _case("square1449_dos", kind=SQUARE, Lx=1449, Ly=1447, W=1.0, S=5, M=1024, nE=2048),
        # local DOS at 32 sites of a disordered cubic lattice
        _case("cubic101_ldos", kind=CUBIC, Lx=101, Ly=103, Lz=99, W=1.5, S=32, sites=True, M=1024, nE=1024),
        # time correlation by concurrent time blocks on vacancy graphene, complex64
        _case("vacancy2048_corr", call="corr", Lx=2048, Ly=2048, t=-2.7, W=2.0, vac=0.01, S=1, Nt=256),
        # the same in complex128
        _case("vacancy1024_corr_c128", call="corr", Lx=1024, Ly=1024, t=-2.7, W=2.0, vac=0.01, c128=True, S=1, Nt=128),
        # DC conductivity of vacancy graphene at 64 energies (quasi-eigenstates, block inner products)
        _case("vacancy1024_dc", call="dc", Lx=1024, Ly=1024, t=-2.7, W=2.0, vac=0.01, S=1, Nt=128, nE=64),
        # optical conductivity of disordered graphene (Fermi-Dirac series, pair propagation)
        _case("graphene1024_optical", call="optical", Lx=1024, Ly=1024, t=-2.7, W=1.0, S=4, Nt=64, nE=1024, kT=0.1),
        # a dense Hamiltonian (234 neighbours per site), DOS from the Fourier form
        _case("dense235_dos", Lx=1832, Ly=1300, t=-2.7, dh=235, S=2, Nt=256, nE=2048, method="fourier"),
        # sixteen requests of different lattices served together (continuous batching and direct lanes)
        _case("serving16", call="serve", mix=7, S=16, M=1024, nE=512),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def even(lo, hi):
        return log(lo, hi) // 2 * 2

    pick = rng.choice(["tiny128", "small", "graphene", "square", "cubic", "vacancy", "vacancy128", "dc", "optical",
                       "dense", "serve"])
    W = round(rng.uniform(0.1, 2.0), 3)
    per = rng.random() < 0.7
    if pick == "tiny128":
        kind = rng.choice([SQUARE, HONEYCOMB])
        return _case(kind=kind, Lx=log(32, 160), Ly=log(32, 160), px=per, W=W, c128=True, S=rng.choice([1, 1, 2, 3]),
                     M=even(256, 1024), nE=log(256, 1024))
    if pick == "small":
        kind = rng.choice([SQUARE, HONEYCOMB, CUBIC])
        L = [log(12, 40) for _ in range(3)] if kind == CUBIC else [log(32, 300), log(32, 300), 1]
        return _case(kind=kind, Lx=L[0], Ly=L[1], Lz=L[2], py=per, W=W, S=rng.randint(1, 16), M=even(256, 1024),
                     nE=log(256, 2048))
    if pick == "graphene":
        return _case(Lx=log(400, 2048), Ly=log(400, 2048), t=-2.7, W=W if rng.random() < 0.7 else 0.0, py=per,
                     S=rng.choice([1, 2, 3, 4, 6, 8]), M=even(256, 2048), nE=log(512, 8192),
                     tensor=rng.random() < 0.5)
    if pick == "square":
        return _case(kind=SQUARE, Lx=log(400, 1449), Ly=log(400, 1449), W=W, px=per, S=rng.randint(1, 8),
                     M=even(256, 1024), nE=log(512, 2048))
    if pick == "cubic":
        sites = rng.random() < 0.5
        return _case(kind=CUBIC, Lx=log(40, 101), Ly=log(40, 101), Lz=log(40, 99), W=W, pz=per, sites=sites,
                     S=32 if sites else rng.randint(1, 16), M=even(256, 1024), nE=log(256, 1024))
    if pick in ("vacancy", "vacancy128"):
        big = pick == "vacancy"
        return _case(call="corr", Lx=log(256, 2048 if big else 1024), Ly=log(256, 2048 if big else 1024), t=-2.7, W=W,
                     vac=round(rng.uniform(0.002, 0.05), 4), c128=not big, S=rng.choice([1, 1, 2]) if big else 1,
                     Nt=log(48, 256 if big else 128))
    if pick == "dc":
        return _case(call="dc", Lx=log(256, 1024), Ly=log(256, 1024), t=-2.7, W=W,
                     vac=round(rng.uniform(0.002, 0.05), 4) if rng.random() < 0.7 else 0.0, S=1, Nt=log(48, 128),
                     nE=log(8, 64))
    if pick == "optical":
        return _case(call="optical", Lx=log(256, 1024), Ly=log(256, 1024), t=-2.7, W=W, S=rng.randint(1, 4),
                     Nt=log(32, 64), nE=log(256, 1024), kT=round(rng.uniform(0.1, 0.4), 3))
    if pick == "dense":
        return _case(Lx=log(300, 1832), Ly=log(300, 1300), t=-2.7, dh=rng.choice([61, 124, 235]), S=2, Nt=log(64, 256),
                     nE=log(512, 2048), method="fourier")
    return _case(call="serve", mix=rng.randint(100, 10**6), S=rng.randint(6, 16), M=even(256, 1024), nE=log(128, 512))


# ---------------------------------------------------------------- requests
_shared = {}


def _ctx():
    """The program's one context, and its server for streams of requests."""
    if "ctx" not in _shared:
        _shared["ctx"] = capi.tbpm_create(0)
    return _shared["ctx"]


def _server():
    if "server" not in _shared:
        _shared["server"] = capi.tbpm_server_create(_ctx())
    return _shared["server"]


def _mix(case, seed):
    """The batch of a serving case: sizes from the case alone, disorder and states from the seed."""
    rng = random.Random(case["mix"])
    seeds = random.Random(seed)
    out = []
    for _ in range(case["S"]):
        kind = rng.randrange(3)
        n = 2.0 ** rng.uniform(12, 18)
        if kind == CUBIC:
            L = [max(4, round(n ** (1 / 3) * f)) for f in (1.0, 1.1, 0.9)]
        else:
            r = math.sqrt(n / (2 if kind == HONEYCOMB else 1))
            L = [max(4, round(r * 1.05)), max(4, round(r / 1.05)), 1]
        sites = rng.random() < 0.25
        out.append(_case(call="dos", kind=kind, Lx=L[0], Ly=L[1], Lz=L[2], W=round(rng.uniform(0.0, 2.0), 3),
                         S=32 if sites else rng.randint(1, 16), sites=sites,
                         M=rng.randint(case["M"] // 4, case["M"]) // 8 * 8, nE=case["nE"],
                         seed=seeds.randrange(1, 1 << 31)))
    return out


def _desc(c, seed):
    return capi.lattice_desc(c["kind"], (c["Lx"], c["Ly"], c["Lz"]), t=c["t"], W=c["W"], vacancy_frac=c["vac"],
                             seed=seed, pbc=(c["px"], c["py"], c["pz"]), cutoff=DENSE_CUTOFF.get(c["dh"], 0.0),
                             decay=DENSE_DECAY if c["dh"] else 0.0)


def _site_list(c, seed, n):
    return np.sort(np.random.default_rng(seed).choice(n, size=c["S"], replace=False)).astype(np.int64)


def _request(c, seed, n):
    kw = {"n_states": c["S"], "precision": capi.C128 if c["c128"] else capi.C64, "state_seed": seed + 1}
    if c["sites"]:
        kw["sites"] = _site_list(c, seed, n)
    if c["call"] == "dos" and c["method"] == "jackson":
        return capi.request(n_moments=c["M"], recon=capi.RECON_TENSOR if c["tensor"] else capi.RECON_FP64, **kw)
    if c["call"] == "dos":
        return capi.request(n_steps=c["Nt"], dos_method=capi.DOS_FOURIER, window=capi.WINDOW_HANN, **kw)
    if c["call"] == "optical":
        return capi.request(form=capi.CONCURRENT_S, n_steps=c["Nt"], window=capi.WINDOW_HANN, **kw)
    return capi.request(form=capi.CONCURRENT_S, n_steps=c["Nt"], **kw)


def _energies(c, H0, half):
    """A midpoint grid over the spectral window (DOS) or its inner 80 % (conductivity)."""
    w = 0.8 * half if c["call"] == "dc" else half
    return H0 - w + 2 * w * (np.arange(c["nE"]) + 0.5) / max(1, c["nE"])


def prepare(case, seed):
    c = case
    if c["call"] == "serve":
        batch = []
        for r in _mix(c, seed):
            H0, half = 0.0, 1.01 * (COORD[r["kind"]] + r["W"] / 2)  # the program's own estimate of the band
            n = r["Lx"] * r["Ly"] * r["Lz"] * (2 if r["kind"] == HONEYCOMB else 1)
            batch.append((_desc(r, r["seed"]), _request(r, r["seed"], n), _energies(r, H0, half)))
        return {"case": c, "server": _server(), "batch": batch}
    ctx = _ctx()
    lat = capi.tbpm_lattice_create(ctx, _desc(c, seed))
    p = capi.tbpm_lattice_info(lat)
    state = _State(case=c, ctx=ctx, lat=lat, req=_request(c, seed, p.n_sites), energies=_energies(c, p.H0, p.half_width))
    weakref.finalize(state, capi.tbpm_lattice_destroy, lat)
    return state


class _State(dict):
    """A request with its lattice handle, which goes with it."""
    __hash__ = object.__hash__


def _kept(c, a):
    """Results in the precision of the request."""
    return a if c["c128"] else a.astype(np.complex64 if np.iscomplexobj(a) else np.float32)


def run(state):
    c = state["case"]
    if c["call"] == "serve":
        srv = state["server"]
        tickets = [capi.tbpm_submit(srv, d, r, e) for d, r, e in state["batch"]]
        out = []
        for t, (_, r, e) in zip(tickets, state["batch"]):
            D = np.empty((r.n_states, e.size))
            capi.tbpm_wait(srv, t, D)
            out.append(_kept(c, D))
        return out
    ctx, lat, req, E = state["ctx"], state["lat"], state["req"], state["energies"]
    if c["call"] == "dos":
        D = np.empty((c["S"], c["nE"]))
        capi.tbpm_dos(ctx, lat, req, E, D)
        return _kept(c, D)
    if c["call"] == "corr":
        C = np.empty((c["S"], c["Nt"] + 1), np.complex128)
        capi.tbpm_correlation(ctx, lat, req, C)
        return _kept(c, C)
    if c["call"] == "dc":
        C = np.empty((c["S"], c["nE"], c["Nt"] + 1), np.complex128)
        sigma = np.empty((c["S"], c["nE"]))
        capi.tbpm_conductivity(ctx, lat, req, 0, E, C, sigma)
        return [_kept(c, C), _kept(c, sigma)]
    C = np.empty((c["S"], c["Nt"] + 1), np.complex128)
    sigma = np.empty((c["S"], c["nE"]), np.complex128)
    capi.tbpm_optical_conductivity(ctx, lat, req, 0, 0, 0.3, c["kT"], 10.0, c["nE"], C, sigma)
    return [_kept(c, C), _kept(c, sigma)]


# ---------------------------------------------------------------- work
def _orders(x):
    """About the number of Chebyshev terms of exp(-i x H~)."""
    return x + 12 * x ** (1 / 3) + 8


def work(case):
    """Floating operations of the recurrence (2 per neighbour and real component for the sum, the
    two scaled additions) and of the inner products and series; bytes of the lattice's arrays, of
    one state block in and out, and of the results.  What a fused pass saves in state traffic is
    not counted as needed."""
    c = case
    if c["call"] == "serve":
        parts = [work({k: v for k, v in r.items() if k != "seed"}) for r in _mix(c, 0)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    z = c["dh"] - 1 if c["dh"] else COORD[c["kind"]]
    N = c["Lx"] * c["Ly"] * c["Lz"] * (2 if c["kind"] == HONEYCOMB else 1) * (1 - c["vac"])
    elem = 16 if c["c128"] else 8
    S, Nt, nE = c["S"], c["Nt"], c["nE"]
    step = (4 * z if c["dh"] else 2 * z) + 8
    lattice = N * ((elem // 2 if c["W"] else 0) + (4 * z if c["vac"] else 0))
    state = 2 * N * S * elem
    if c["call"] == "dos":
        M = c["M"] if c["method"] == "jackson" else _orders(Nt * math.pi)
        return {"bytes": lattice + state + 8 * nE * (S + 1), "flops": N * S * (M / 2) * (step + 8) + 4.0 * M * nE * S}
    if c["call"] == "corr":
        blocks = max(1, Nt // 16)
        per = _orders(16 * math.pi)
        adds = sum(_orders(j * math.pi) for j in range(1, 17)) * blocks
        return {"bytes": lattice + state, "flops": N * S * (blocks * per * step + adds * 8 + 8 * Nt)}
    if c["call"] == "dc":
        qe = _orders(Nt * math.pi)
        prop = max(1, Nt // 16) * _orders(16 * math.pi)
        adds = sum(_orders(j * math.pi) for j in range(1, 17)) * max(1, Nt // 16)
        return {"bytes": lattice + state * nE, "flops": N * S * ((qe + prop) * step + 4 * qe * nE + 8 * adds + 8 * Nt * nE)}
    fermi = 12 * 1.01 * (3 * 2.7 + c["W"] / 2) / c["kT"]
    prop = max(1, Nt // 16) * _orders(8 * math.pi)
    adds = sum(_orders(j * math.pi / 2) for j in range(1, 17)) * max(1, Nt // 16)
    return {"bytes": lattice + 2 * state, "flops": 2 * N * S * ((fermi + prop) * step + 4 * fermi + 8 * adds + 8 * Nt)}


# ---------------------------------------------------------------- the same in 64 bits
_DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _draw32(seed, idx, stream, sub):
    """First word of Philox4x32-10 at counter (idx, stream, sub), as int64."""
    m = 0xFFFFFFFF

    def mul(a, c):
        p, q = (c & 0xFFFF) * a, (c >> 16) * a
        s = q + (p >> 16)
        return s >> 16, ((s & 0xFFFF) << 16) | (p & 0xFFFF)

    c0, c1 = idx & m, idx >> 32
    c2, c3 = torch.full_like(idx, stream), torch.full_like(idx, sub)
    k0, k1 = seed & m, (seed >> 32) & m
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c0


class _Lat:
    """A lattice's neighbour lists, on-site energies and bounds, for nearest neighbours."""

    def __init__(self, c, seed):
        kind, Lx, Ly, Lz = c["kind"], c["Lx"], c["Ly"], c["Lz"]
        n = Lx * Ly * Lz * (2 if kind == HONEYCOMB else 1)
        i = torch.arange(n, device=_DEV)
        s = i % 2 if kind == HONEYCOMB else torch.zeros(1, dtype=torch.int64, device=_DEV)
        q = i // 2 if kind == HONEYCOMB else i
        x, y, z = q % Lx, (q // Lx) % Ly, q // (Lx * Ly)
        sg = 2 * s - 1
        step = {SQUARE: [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0)],
                CUBIC: [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)],
                HONEYCOMB: [(0, 0, 0), (1, 0, 0), (0, 1, 0)]}[kind]
        active = torch.ones(n, dtype=torch.bool, device=_DEV)
        if c["vac"]:
            active = _draw32(seed, i, 1, 0) >= int(math.floor(c["vac"] * 2.0**32))
        self.full = torch.nonzero(active).flatten() if c["vac"] else i
        self.n = self.full.numel()
        compact = torch.cumsum(active, 0) - 1 if c["vac"] else None
        self.nbr = []
        deg = torch.zeros(self.n, device=_DEV, dtype=torch.float64)
        for dx, dy, dz in step:
            if kind == HONEYCOMB:
                dx, dy = dx * sg, dy * sg
            tx, ty, tz = x + dx, y + dy, z + dz
            ok = torch.ones(n, dtype=torch.bool, device=_DEV)
            for v, L, p in ((tx, Lx, c["px"]), (ty, Ly, c["py"]), (tz, Lz, c["pz"])):
                if not p:
                    ok &= (v >= 0) & (v < L)
            tx, ty, tz = tx % Lx, ty % Ly, tz % Lz
            j = 2 * (ty * Lx + tx) + (1 - s) if kind == HONEYCOMB else (tz * Ly + ty) * Lx + tx
            ok &= active[j]
            if c["vac"]:
                ok, j = ok[self.full], compact[j][self.full]
            deg += ok
            self.nbr.append((torch.where(ok, j, 0).to(torch.int32), None if bool(ok.all()) else ok.double()[:, None]))
        del i, q, x, y, z, active, compact
        self.V = None
        v = torch.zeros(1, dtype=torch.float64, device=_DEV)
        if c["W"]:
            v = c["W"] * ((_draw32(seed, self.full, 0, 0) >> 8).double() * 2.0**-24 - 0.5)
            self.V = v[:, None]
        e1, e0 = float((v + deg * abs(c["t"])).max()), float((v - deg * abs(c["t"])).min())
        self.t, self.H0, self.half = c["t"], (e1 + e0) / 2, 1.01 * (e1 - e0) / 2
        self.sub = (self.full % 2).bool() if kind == HONEYCOMB else None
        self.kind = kind

    def H(self, x):
        """(H - H0)/|H| x for complex x [n, S]."""
        r = torch.zeros_like(x)
        for j, ok in self.nbr:
            g = torch.index_select(x, 0, j)
            if ok is not None:
                torch.view_as_real(g).mul_(ok[:, :, None])
            r += g
            del g
        r = torch.view_as_real(r).mul_(self.t / self.half)
        xr = torch.view_as_real(x)
        d = -self.H0 / self.half if self.V is None else ((self.V - self.H0) / self.half)[:, :, None]
        return torch.view_as_complex(r.addcmul_(xr, torch.as_tensor(d, dtype=torch.float64, device=_DEV)))

    def series(self, x, n):
        """T_0 x, T_1 x, ..., n of them."""
        a = x
        yield a
        if n > 1:
            b = self.H(x)
            yield b
        for _ in range(n - 2):
            h = self.H(b)
            torch.view_as_real(h).mul_(2.0)
            h -= a
            a, b = b, h
            yield b

    def current_x(self, x):
        """J_x x with J_ij = -i t (r_j - r_i)_x."""
        w = {HONEYCOMB: (1.0, -0.5, -0.5), SQUARE: (1, -1, 0, 0), CUBIC: (1, -1, 0, 0, 0, 0)}[self.kind]
        r = torch.zeros_like(x)
        for (j, ok), f in zip(self.nbr, w):
            if f:
                g = torch.index_select(x, 0, j)
                r += f * (g if ok is None else g * ok)
        if self.sub is not None:
            r = torch.where(self.sub[:, None], -r, r)
        return -1j * self.t * r

    def states(self, c, seed):
        if c["sites"]:
            x = torch.zeros(self.n, c["S"], dtype=torch.complex128, device=_DEV)
            x[torch.from_numpy(_site_list(c, seed, self.n)).to(_DEV), torch.arange(c["S"], device=_DEV)] = 1.0
            return x
        x = torch.empty(self.n, c["S"], dtype=torch.complex128, device=_DEV)
        for s in range(c["S"]):
            u = _draw32(seed + 1, self.full, 2, s).double() * (math.pi * 2.0**-31)
            x[:, s] = torch.complex(torch.cos(u), torch.sin(u)) / math.sqrt(self.n)
        return x


def _dots(a, b):
    """<a_s|b_s> of every column."""
    return (a.conj() * b).sum(0)


def _moments(lat, x, M):
    """m_n of every state, [S, M], from M/2 products with H."""
    m = torch.empty(M, x.shape[1], dtype=torch.complex128, device=_DEV)
    last = None
    for n, p in enumerate(lat.series(x, M // 2 + 1)):
        if n < M // 2:
            m[2 * n] = _dots(p, p) * (1 if n == 0 else 2) - (0 if n == 0 else m[0])
        if n:
            m[2 * n - 1] = _dots(p, last) * (1 if n == 1 else 2) - (0 if n == 1 else m[1])
        last = p
    return m.T


def _clean_bands(c):
    """Energies of a clean periodic honeycomb at every k point and band (tensor [2, Ly, Lx]), and the phase of
    its sublattice coupling: T(k) couples A to B, H(k) = [[g, f], [f*, g]]."""
    Lx, Ly = c["Lx"], c["Ly"]
    f = torch.zeros(Ly, Lx, dtype=torch.complex128)
    g = torch.zeros(Ly, Lx, dtype=torch.complex128)
    taps = [(0, 0, 1, 1.0), (-1, 0, 1, 1.0), (0, -1, 1, 1.0)]
    if c["dh"]:
        cut, taps = DENSE_CUTOFF[c["dh"]], []
        R = math.ceil(cut) + 2
        for dy in range(-R, R + 1):
            for dx in range(-R, R + 1):
                for ds in (0, 1):
                    r2 = (1.5 * (dx + dy) + ds) ** 2 + 0.75 * (dx - dy) ** 2
                    if 0 < r2 <= cut * cut:
                        taps.append((dx, dy, ds, math.exp(-(math.sqrt(r2) - 1) / DENSE_DECAY)))
    for dx, dy, ds, w in taps:  # (H psi)_A(r) = sum w psi_ds(r + d): in k space the conjugate kernel
        (f if ds else g)[-dy % Ly, -dx % Lx] += w * c["t"]
    f, g = torch.fft.fft2(f.to(_DEV)), torch.fft.fft2(g.to(_DEV)).real
    rad = abs(c["t"]) * sum(w for _, _, _, w in taps)
    return torch.stack([g + f.abs(), g - f.abs()]), torch.angle(f), 1.01 * rad


def _clean_weights(c, seed, phase):
    """|<k, band|psi_s>|^2 of the random states, [S, 2, Ly, Lx]."""
    n = 2 * c["Lx"] * c["Ly"]
    i = torch.arange(n, device=_DEV)
    out = torch.empty(c["S"], 2, c["Ly"], c["Lx"], dtype=torch.float64, device=_DEV)
    rot = torch.polar(torch.ones_like(phase), phase)
    for s in range(c["S"]):
        u = _draw32(seed + 1, i, 2, s).double() * (math.pi * 2.0**-31)
        x = (torch.complex(torch.cos(u), torch.sin(u)) / math.sqrt(n)).view(c["Ly"], c["Lx"], 2)
        a, b = torch.fft.fft2(x[..., 0]), torch.fft.fft2(x[..., 1])
        b = rot * b
        k = 1 / math.sqrt(2 * c["Lx"] * c["Ly"])
        out[s, 0], out[s, 1] = ((a + b) * k).abs().square(), ((a - b) * k).abs().square()
    return out


def _cheb(f, n):
    """Chebyshev coefficients a_0 .. a_{n-1} of the functions f(x) -> [rows, nodes], exact to rounding."""
    K = 2 * n + 64
    th = math.pi * (np.arange(K) + 0.5) / K
    v = np.atleast_2d(f(np.cos(th)))
    F = np.fft.fft(np.concatenate([v, v[:, ::-1]], axis=1), axis=1)[:, :n]
    a = F * np.exp(-0.5j * math.pi * np.arange(n) / K) / K
    a[:, 0] *= 0.5
    return a


def _evolution(taus, n):
    """c_n of exp(-i x tau) for every tau, [taus, n]."""
    return _cheb(lambda x: np.exp(-1j * np.outer(taus, x)), n)


def _jackson(m, E, H0, half):
    S, M = m.shape
    n = torch.arange(M, device=_DEV, dtype=torch.float64)
    q = math.pi / (M + 1)
    g = ((M - n + 1) * torch.cos(q * n) + torch.sin(q * n) / math.tan(q)) / (M + 1) * torch.where(n == 0, 1.0, 2.0)
    x = (torch.from_numpy(E).to(_DEV) - H0) / half
    ok = x.abs() < 1
    th = torch.acos(x.clamp(-1, 1))
    D = (m.real * g) @ torch.cos(n[:, None] * th)
    return torch.where(ok, D / (math.pi * half * torch.sqrt((1 - x * x).clamp_min(1e-300))), 0.0)


def _window(Nt):
    return 0.5 * (1 + np.cos(math.pi * np.arange(Nt + 1) / (Nt + 1.0)))


def _fourier(C, E, tau):
    Nt = C.shape[1] - 1
    w = _window(Nt) * np.where(np.arange(Nt + 1) == 0, 1.0, 2.0)
    return tau / (2 * math.pi) * ((w * C) @ np.exp(1j * np.outer(np.arange(Nt + 1) * tau, E))).real


def _exact_dos(c, seed, energies=None):
    if c["W"] == 0 and c["kind"] == HONEYCOMB and c["px"] and c["py"] and not c["sites"] and not c["vac"]:
        E, phase, half = _clean_bands(c)
        w = _clean_weights(c, seed, phase).reshape(c["S"], -1)
        e = E.reshape(-1)
        if c["method"] == "fourier":
            C = np.empty((c["S"], c["Nt"] + 1), np.complex128)
            for j in range(c["Nt"] + 1):
                u = e * (j * math.pi / half)
                C[:, j] = (w @ torch.cos(u) - 1j * (w @ torch.sin(u))).cpu().numpy()
            return _fourier(C, _energies(c, 0.0, half), math.pi / half)
        x = e / half
        m = torch.empty(c["S"], c["M"], dtype=torch.float64, device=_DEV)
        a, b = torch.ones_like(x), x.clone()
        for n in range(c["M"]):
            m[:, n] = w @ a
            a, b = b, torch.addcmul(-a, x, b, value=2.0)
        return _jackson(m, _energies(c, 0.0, half) if energies is None else energies, 0.0, half)
    lat = _Lat(c, seed)
    m = _moments(lat, lat.states(c, seed), c["M"])
    return _jackson(m, _energies(c, lat.H0, lat.half) if energies is None else energies, lat.H0, lat.half)


def _exact_corr(c, seed):
    lat = _Lat(c, seed)
    taus = math.pi * np.arange(c["Nt"] + 1)
    M = int(_orders(taus[-1])) // 2 * 2 + 40
    m = _moments(lat, lat.states(c, seed), M).cpu().numpy()
    return (m @ _evolution(taus, M).T) * np.exp(-1j * lat.H0 / lat.half * taus)


def _exact_dc(c, seed):
    lat = _Lat(c, seed)
    psi = lat.states(c, seed)
    E, Nt = _energies(c, lat.H0, lat.half), c["Nt"]
    taus, tau = math.pi * np.arange(Nt + 1), math.pi / lat.half
    n = int(_orders(taus[-1])) + 40

    def line(x):  # (tau/2pi) sum_{|j| <= Nt} e^{i (E - H0 - |H| x) t_j}
        d = (E[:, None] - lat.H0) / lat.half - x[None, :]
        s = np.ones_like(d)
        for t in taus[1:]:
            s += 2.0 * np.cos(d * t)
        return tau / (2 * math.pi) * s

    coef = torch.from_numpy(_cheb(line, n).real).to(_DEV)
    sigma, C = np.empty((c["S"], c["nE"])), np.empty((c["S"], c["nE"], Nt + 1), np.complex128)
    area = 3 * SQ3 / 4 if c["kind"] == HONEYCOMB else 1.0
    for s in range(c["S"]):
        x = psi[:, s:s + 1]
        qe = torch.zeros(lat.n, c["nE"], dtype=torch.complex128, device=_DEV)
        flat = torch.view_as_real(qe)
        for k, p in enumerate(lat.series(x, n)):
            flat += torch.view_as_real(p) * coef[:, k][None, :, None]
        o = (x.conj() * qe).sum(0).cpu().numpy()
        for k in range(c["nE"]):
            qe[:, k] = lat.current_x(qe[:, k:k + 1])[:, 0]
        m = torch.empty(n, c["nE"], dtype=torch.complex128, device=_DEV)
        for k, p in enumerate(lat.series(lat.current_x(x), n)):
            m[k] = (p.conj().T @ qe)[0]
        ev = np.conj(_evolution(taus, n)) * np.exp(1j * lat.H0 / lat.half * taus)[:, None]
        C[s] = (ev @ m.cpu().numpy()).T / np.abs(o)[:, None]
        w = np.where(np.arange(Nt + 1) == 0, 0.5, 1.0)
        tj = tau * np.arange(Nt + 1)
        sigma[s] = o.real / area * tau * (w * np.exp(-1j * np.outer(E, tj)) * C[s]).real.sum(1)
    return [C, sigma]


def _exact_optical(c, seed):
    lat = _Lat(c, seed)
    psi = lat.states(c, seed)
    jpsi = lat.current_x(psi)
    S, Nt, kT, K = c["S"], c["Nt"], c["kT"], c["nE"]
    nf = int(min(16384, 12 * lat.half / kT + 64))
    fermi = _cheb(lambda x: 0.5 * (1 - np.tanh((lat.H0 + lat.half * x - 0.3) / (2 * kT))), nf).real[0]
    X = torch.cat([psi, jpsi], 1)
    F = torch.zeros_like(X)
    for a, p in zip(fermi, lat.series(X, nf)):
        F.add_(p, alpha=float(a))
    Y = torch.cat([F[:, :S], jpsi - F[:, S:]], 1)
    n = int(_orders(math.pi / 2)) + 30
    ev = _evolution([math.pi / 2], n)[0]
    C = np.empty((S, Nt + 1), np.complex128)
    for j in range(Nt + 1):
        C[:, j] = _dots(Y[:, :S], lat.current_x(Y[:, S:])).cpu().numpy()
        if j < Nt:
            Z = torch.zeros_like(Y)
            for a, p in zip(ev, lat.series(Y, n)):
                Z.add_(p, alpha=complex(a))
            Y = Z
    tau, area = math.pi / 2 / lat.half, 3 * SQ3 / 4
    om = np.arange(K) * (10.0 / (K - 1))
    w = _window(Nt) * np.where(np.arange(Nt + 1) == 0, 0.5, 1.0)
    kernel = np.sin(np.outer(om, tau * np.arange(Nt + 1)))
    re = np.zeros((S, K))
    re[:, 1:] = 2 * np.expm1(-om[1:] / kT) / (om[1:] * area) * tau * ((w * C.imag) @ kernel.T)[:, 1:]
    k = np.arange(K)
    odd = (k[:, None] - k[None, :]) % 2 == 1
    den = np.where(odd, om[None, :] ** 2 - om[:, None] ** 2, 1.0)
    wq = np.where(odd, np.where(k == 0, 1.0, 2.0)[None, :] * om[1] / den, 0.0)
    im = -(2 * om / math.pi) * (re @ wq.T)
    return [C, re + 1j * im]


def exact(case, seed):
    c = case
    if c["call"] == "serve":
        out = []
        for r in _mix(c, seed):
            half = 1.01 * (COORD[r["kind"]] + r["W"] / 2)
            out.append(_exact_dos(r, r["seed"], _energies(r, 0.0, half)))
        return out
    return {"dos": _exact_dos, "corr": _exact_corr, "dc": _exact_dc, "optical": _exact_optical}[c["call"]](c, seed)
