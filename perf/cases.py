"""Performance cases: the work a user of this framework has it do, through its public calls.

Every case is one call of the torch front end (`paper_2506_09551_gb300.api`) on inputs that
a program already holds on the device: an operator apply, a ground state, a multi-shift
solve, a batch of continued fractions, or a whole RIXS map.  Sizes are those of the named
workloads (chains of 8 to 14 sites, 41 to 201 incident energies, a random symmetric matrix
with about 16 entries per row) and of the tests, with open chains, odd fillings and periodic
2D clusters with diagonal hopping among the drawn ones.

`exact` recomputes a case in 64 bits with plain torch and numpy: Hamiltonians from the
bit-string definition (dense blocks of one spin species), Lanczos, conjugate-orthogonal
conjugate gradients and the Lehmann sum.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2506_09551_gb300 import api

T, U, UC = 1.0, 8.0, 4.0          # hopping, repulsion and core-hole potential of the workloads
GAMMA, ETA = 0.3, 0.1             # inverse core-hole lifetime and loss broadening
E_SITE = -0.33                    # ground-state energy per site of the half-filled chain at U = 8


def _case(name, kind, **kw):
    c = dict(name=name, kind=kind, L=0, nu=0, nd=0, ring=True, lx=0, tp=0.0, mixed=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one product with H' on a six-site ring, as in a small-cluster
        # study or a user's own iteration; launch latency decides
        _case("apply-L6", "apply", L=6, nu=4, nd=3, core=True, nvec=1),
        # a block of FP64 vectors through H at the size of the 12-site workload
        _case("apply-L12-block", "apply", L=12, nu=6, nd=6, core=False, nvec=8),
        # the largest sector, FP32: one product with H' of the 14-site ring
        _case("apply-L14-mixed", "apply", L=14, nu=8, nd=7, core=True, nvec=1, mixed=True),
        # |G> and E_G of the 12-site ring, the first step of every map (FP64 in every mode)
        _case("ground-L12", "ground", L=12, nu=6, nd=6),
        # the 8-site workload's solve for c^dag|G>: 41 incident energies, a latency-bound recurrence
        _case("solve-L8", "solve", L=8, nu=5, nd=4, shifts=41, tol=1e-12, iters=1140),
        # the 12-site workload's solve in FP64 to a tight tolerance
        _case("solve-L12", "solve", L=12, nu=7, nd=6, shifts=41, tol=1e-12, iters=1700),
        # a 13-site sector (rows of odd parity in L, signed hops) in the FP32-mixed form
        _case("solve-L13-mixed", "solve", L=13, nu=7, nd=6, shifts=48, tol=1e-8, iters=1320, mixed=True),
        # the random symmetric matrix with many shifts, FP64, a size that is no power of two
        _case("solve-csr", "csr", n=200003, half=8, shifts=128, tol=1e-11, iters=1000),
        # second step of the 12-site map in FP64: some columns, a fixed number of levels
        _case("cf-L12", "cf", L=12, nu=6, nd=6, nvec=24, depth=60, n_w=400),
        # second step of the 14-site map in FP32
        _case("cf-L14-mixed", "cf", L=14, nu=7, nd=7, nvec=8, depth=48, n_w=400, mixed=True),
        # a whole small map in FP64 with the default parameters (the 8-site workload)
        _case("map-L8", "map", L=8, nu=4, nd=4, n_in=41, n_w=200),
        # a whole batch in FP32: the maps of all core sites of a 10-site ring in one call
        _case("sites-L10-mixed", "sites", L=10, nu=5, nd=5, n_in=16, n_w=400, mixed=True),
    ]


def _dim(L, nu, nd):
    return math.comb(L, nu) * math.comb(L, nd)


def _lattice(rng, c, small):
    """A ring, an open chain or a periodic 3 x 3 / 3 x 4 cluster with or without t'."""
    r = rng.random()
    if r < 0.2:
        L = 9 if small or rng.random() < 0.5 else 12
        c.update(L=L, lx=3, tp=rng.choice([0.0, -0.3, 0.2]))
    else:
        c.update(L=rng.randint(4, 10 if small else 13), ring=rng.random() < 0.7)
    return c


def draw(rng):
    kind = rng.choice(["apply", "apply", "solve", "solve", "cf", "cf", "csr", "ground", "map"])
    mixed = rng.random() < 0.5
    c = _case("", kind, mixed=mixed)
    del c["name"]
    if kind == "apply":
        _lattice(rng, c, False)
        c.update(nu=rng.randint(1, c["L"] - 1), nd=rng.randint(1, c["L"] - 1), core=rng.random() < 0.5)
        most = max(1, min(16, 8_000_000 // _dim(c["L"], c["nu"], c["nd"])))
        c.update(nvec=rng.randint(1, most))
    elif kind == "solve":
        _lattice(rng, c, True)
        c.update(nu=rng.randint(2, c["L"] - 1), nd=rng.randint(1, c["L"] - 1),
                 shifts=int(round(math.exp(rng.uniform(0.0, math.log(64))))), tol=1e-8 if mixed else 1e-12, iters=900)
    elif kind == "cf":
        _lattice(rng, c, False)
        c.update(nu=rng.randint(1, c["L"] - 1), nd=rng.randint(1, c["L"] - 1), n_w=rng.randint(20, 400))
        D = _dim(c["L"], c["nu"], c["nd"])
        c.update(depth=min(rng.randint(16, 60), max(2, D // 8)))
        c.update(nvec=rng.randint(1, max(1, min(32, 20_000_000 // D))))
    elif kind == "csr":
        # FP64 only: the FP32 solutions of the random matrix are themselves 1e-5 off
        c.update(mixed=False, n=int(round(math.exp(rng.uniform(math.log(2000), math.log(200003))))), half=rng.randint(4, 10),
                 shifts=int(round(math.exp(rng.uniform(0.0, math.log(128))))), tol=1e-11, iters=1000)
    elif kind == "ground":
        # unique ground states: open chains at any filling, half-filled even rings
        if rng.random() < 0.5:
            L = rng.randint(4, 12)
            c.update(L=L, ring=False, nu=rng.randint(1, L - 1), nd=rng.randint(1, L - 1), mixed=False)
        else:
            L = rng.choice([4, 6, 8, 10, 12])
            c.update(L=L, nu=L // 2, nd=L // 2, mixed=False)
    else:
        L = rng.randint(4, 8)
        c.update(L=L, ring=False, nu=rng.randint(1, L - 1), nd=rng.randint(1, L - 1), n_in=rng.randint(3, 41),
                 n_w=rng.randint(20, 200))
    return c


# ---------------------------------------------------------------------------
# what a program holds before the call
# ---------------------------------------------------------------------------
def _cdtype(c):
    return torch.complex64 if c["mixed"] else torch.complex128


def _prec(c):
    return api.FP32_MIXED if c["mixed"] else api.FP64


def _vectors(c, seed, nvec, dim):
    """Random complex vectors with N(0, 1) parts, drawn in 64 bits and rounded to the case's precision."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 17)
    x = torch.empty((nvec, dim), dtype=_cdtype(c), device="cuda")
    for k in range(nvec):
        re = torch.randn(dim, generator=g, dtype=torch.float64, device="cuda")
        im = torch.randn(dim, generator=g, dtype=torch.float64, device="cuda")
        x[k] = torch.complex(re, im).to(_cdtype(c))
    return x


def _couplings(c, seed):
    """U and U_c near the workloads' values, another pair for each seed."""
    r = np.random.RandomState(seed % (1 << 31))
    return U + r.uniform(-0.5, 0.5), UC + r.uniform(-0.25, 0.25)


def _grids(c):
    return np.linspace(-4.0, 12.0, c.get("n_in", 1)), np.linspace(-1.0, 10.0, c.get("n_w", 1))


def _model(c, u=U, uc=UC, inter=False):
    """The model whose ground sector is (nu, nd), or whose intermediate sector is."""
    return api.model(c["L"], c["nu"] - (1 if inter else 0), c["nd"], t=T, U=u, Uc=uc, core_site=0,
                     periodic=bool(c["ring"]), lx=c["lx"], tp=c["tp"])


def _csr(c, seed):
    """Random real symmetric matrix, `half` drawn columns per row mirrored, in CSR form (numpy)."""
    n, h = c["n"], c["half"]
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 29)
    rows = torch.arange(n, device="cuda").repeat_interleave(h)
    cols = torch.randint(0, n - 1, (n * h,), generator=g, device="cuda")
    cols = cols + (cols >= rows)
    vals = torch.randn(n * h, generator=g, dtype=torch.float64, device="cuda")
    diag = torch.rand(n, generator=g, dtype=torch.float64, device="cuda") * 8.0 - 4.0
    d = torch.arange(n, device="cuda")
    key = torch.cat([rows * n + cols, cols * n + rows, d * n + d])
    val = torch.cat([vals, vals, diag])
    key, order = torch.sort(key, stable=True)
    key, val = key.cpu().numpy(), val[order].cpu().numpy()
    uniq, start = np.unique(key, return_index=True)
    val = np.add.reduceat(val, start)
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(uniq // n, minlength=n))]).astype(np.int64)
    return rowptr, (uniq % n).astype(np.int32), val


def _csr_shifts(c, seed):
    """Shifts with real parts spread over [-6, 6] and width 0.3; the middle one is the seed system."""
    r = np.random.RandomState((seed + 7) % (1 << 31))
    sig = np.sort(r.uniform(-6.0, 6.0, c["shifts"])) + 0.3j
    s0 = sig[len(sig) // 2]
    return s0, sig - s0


def _rhs(c, seed):
    """b = c^dag_{0,up}|G> in the case's sector (nu, nd) as a complex vector, and E_G: the ground state of
    (nu - 1, nd) by a plain Lanczos run (any vector close to it serves as the right-hand side)."""
    u, uc = _couplings(c, seed)
    lo = dict(c, nu=c["nu"] - 1)
    H = _hamiltonian(lo, False, u, uc)
    D = _dim(c["L"], lo["nu"], c["nd"])
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 41)
    v = torch.randn(D, generator=g, dtype=torch.float64, device="cuda")
    Q, a, b = [v / torch.linalg.vector_norm(v)], [], []
    for k in range(min(D, 80)):
        y = H(Q[-1][:, None])[:, 0]
        a.append(float(torch.dot(Q[-1], y)))
        y = y - a[-1] * Q[-1] - (b[-1] * Q[-2] if k else 0.0)
        b.append(float(torch.linalg.vector_norm(y)))
        if b[-1] < 1e-10:
            break
        Q.append(y / b[-1])
    m = len(a)
    E, Y = np.linalg.eigh(np.diag(a) + np.diag(b[:m - 1], 1) + np.diag(b[:m - 1], -1))
    G = sum(float(Y[k, 0]) * Q[k] for k in range(m)).reshape(-1, math.comb(c["L"], c["nd"]))
    src, dst = _created(c["L"], c["nu"] - 1)
    out = torch.zeros((math.comb(c["L"], c["nu"]), G.shape[1]), dtype=torch.float64, device="cuda")
    out[dst] = G[src]
    return out.reshape(-1).to(_cdtype(c)), float(E[0])


def _solve_system(c, E):
    """Seed system and shifts of an incident grid on [-4, 12], seeded next to the atomic resonance."""
    w = np.linspace(-4.0, 12.0, c["shifts"]) if c["shifts"] > 1 else np.array([0.7])
    s0 = w[int(np.argmin(np.abs(w)))]
    return complex(-E - s0, -GAMMA), (w - s0).astype(np.complex128)


def prepare(case, seed):
    c = dict(case)
    s = {"case": c}
    kind = c["kind"]
    if kind == "apply":
        s["op"] = api.Operator.hubbard(_model(c, inter=c["core"]), c["core"])
        s["x"] = _vectors(c, seed, c["nvec"], s["op"].dim)
    elif kind == "solve":
        s["op"] = api.Operator.hubbard(_model(c, *_couplings(c, seed), inter=True), True)
        s["b"], E = _rhs(c, seed)
        s["c0"], s["shifts"] = _solve_system(c, E)
    elif kind == "csr":
        s["op"] = api.Operator.csr(*_csr(c, seed))
        s["b"] = _vectors(c, seed, 1, c["n"])[0]
        s0, s["shifts"] = _csr_shifts(c, seed)
        s["c0"] = -s0
    elif kind == "cf":
        s["op"] = api.Operator.hubbard(_model(c))
        s["phi"] = _vectors(c, seed, c["nvec"], s["op"].dim)
        s["w"] = _grids(c)[1]
    elif kind == "ground":
        u, uc = _couplings(c, seed)
        s["op"] = api.Operator.hubbard(_model(c, u, uc))
    else:
        u, uc = _couplings(c, seed)
        s["model"] = _model(c, u, uc)
        s["w_in"], s["w"] = _grids(c)
        tol = dict(solve_tol=1e-8, cf_tol=1e-6) if c["mixed"] else {}
        s["params"] = api.map_params(Gamma=GAMMA, eta=ETA, precision=_prec(c), **tol)
        s["sites"] = list(range(c["L"]))
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _kept(c, I):
    """Intensities as a program keeps them: in the precision of the vectors they were computed from."""
    return I.astype(np.float32) if c["mixed"] else I


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "apply":
        return s["op"].apply(s["x"], complex(0.33 * c["L"], -GAMMA))
    if kind in ("solve", "csr"):
        x, per, _, _ = s["op"].multishift_solve(s["b"], s["shifts"], s["c0"], tol=c["tol"], maxit=5000, prec=_prec(c))
        return {"x": x, "converged": per["converged"]}
    if kind == "cf":
        I, depth = s["op"].continued_fraction(s["phi"], E_SITE * c["L"], s["w"], ETA, cf_tol=0.0, cf_check=c["depth"],
                                              cf_maxdepth=c["depth"])
        return {"I": _kept(c, I), "depth": depth}
    if kind == "ground":
        E, g, _ = s["op"].ground_state(1e-12, 300)
        return {"E": E, "g": g}
    if kind == "map":
        I, info, _ = api.rixs_map(s["model"], s["params"], s["w_in"], s["w"])
        return {"I": _kept(c, I), "E": info["E_G"]}
    I, info, _ = api.rixs_map_sites(s["model"], s["params"], s["sites"], s["w_in"], s["w"])
    return {"I": _kept(c, I), "E": info["E_G"]}


def work(case):
    c = case
    cb = 8.0 if c["mixed"] else 16.0
    if c["kind"] == "csr":
        n, nnz = c["n"], c["n"] * (2 * c["half"] + 1)
        it = c["iters"]
        return {"bytes": nnz * (4 + cb / 2) + n * cb * (1 + c["shifts"]),
                "flops": it * (4.0 * nnz + 28.0 * n + 16.0 * n * c["shifts"])}
    L, D = c["L"], _dim(c["L"], c["nu"], c["nd"])
    bonds = (L if c["ring"] else L - 1) if not c["lx"] else (2 * L + (2 * L if c["tp"] else 0))
    hops = 2 * bonds * sum(k * (L - k) for k in (c["nu"], c["nd"])) / (L * (L - 1.0))   # mean per state
    hx = D * (2.0 * hops + 6.0)                            # one complex product
    if c["kind"] == "apply":
        return {"bytes": 2 * cb * D * c["nvec"], "flops": c["nvec"] * (hx + 8.0 * D)}
    if c["kind"] == "solve":
        return {"bytes": cb * D * (1 + c["shifts"]),
                "flops": c["iters"] * (hx + 36.0 * D + 16.0 * D * c["shifts"])}
    if c["kind"] == "cf":
        return {"bytes": cb * D * c["nvec"] + 8.0 * c["nvec"] * c["n_w"],
                "flops": c["nvec"] * c["depth"] * (hx + 20.0 * D)}
    if c["kind"] == "ground":
        return {"bytes": 8.0 * D, "flops": 100 * (hx / 2 + 10.0 * D)}
    cols = c["n_in"] * (L if c["kind"] == "sites" else 1)
    depth = min(D, 60 * L)
    return {"bytes": 8.0 * cols * c["n_w"], "flops": cols * depth * (hx + 20.0 * D) + 500.0 * 16.0 * D * cols}


# ---------------------------------------------------------------------------
# the same in 64 bits, from the definitions
# ---------------------------------------------------------------------------
def _states(L, n):
    return [sum(1 << i for i in s) for s in sorted(itertools.combinations(range(L), n), key=lambda s: sum(1 << i for i in s))]


def _created(L, n):
    """Ranks of the n-electron strings without site 0, and of the same strings with it (no electron
    of the species sits below site 0: the operator's sign is +)."""
    lo, hi = _states(L, n), {s: i for i, s in enumerate(_states(L, n + 1))}
    src = [i for i, s in enumerate(lo) if not s & 1]
    return torch.tensor(src, device="cuda"), torch.tensor([hi[lo[i] | 1] for i in src], device="cuda")


def _bonds(c):
    L, lx = c["L"], c["lx"]
    if not lx:
        return [(i, (i + 1) % L, T) for i in range(L if c["ring"] else L - 1)]
    ly, out = L // lx, []
    site = lambda x, y: x % lx + lx * (y % ly)  # noqa: E731
    for y in range(ly):
        for x in range(lx):
            out += [(site(x, y), site(x + 1, y), T), (site(x, y), site(x, y + 1), T)]
            if c["tp"]:
                out += [(site(x, y), site(x + 1, y + 1), c["tp"]), (site(x, y), site(x - 1, y + 1), c["tp"])]
    return out


def _hopping(c, n):
    """-sum t c^dag c of one spin species as a sparse matrix, and the occupation strings."""
    st = _states(c["L"], n)
    rank = {s: i for i, s in enumerate(st)}
    r, q, v = [], [], []
    for i, j, t in _bonds(c):
        a, b = min(i, j), max(i, j)
        between = ((1 << b) - 1) ^ ((1 << (a + 1)) - 1)
        for s in st:
            if ((s >> i) & 1) != ((s >> j) & 1):
                r.append(rank[s])
                q.append(rank[s ^ (1 << i) ^ (1 << j)])
                v.append(-t * (-1.0) ** bin(s & between).count("1"))
    m = torch.sparse_coo_tensor(torch.tensor([r, q], dtype=torch.int64).reshape(2, -1), torch.tensor(v, dtype=torch.float64),
                                (len(st), len(st)), device="cuda").coalesce()
    return m, np.array(st, dtype=np.int64)


def _hamiltonian(c, core, u=U, uc=UC):
    """x -> H x for a block of real FP64 columns x of shape (D, m)."""
    Tu, su = _hopping(c, c["nu"])
    Td, sd = _hopping(c, c["nd"])
    both = su[:, None] & sd[None, :]
    pop = sum((both >> i) & 1 for i in range(c["L"]))
    diag = u * pop - (uc * ((su & 1)[:, None] + (sd & 1)[None, :]) if core else 0.0)
    diag = torch.tensor(diag, dtype=torch.float64, device="cuda").reshape(-1, 1)
    Du, Dd = len(su), len(sd)

    def H(x):
        m = x.shape[1]
        up = torch.sparse.mm(Tu, x.reshape(Du, Dd * m)).reshape(Du * Dd, m)
        dn = x.reshape(Du, Dd, m).permute(1, 0, 2).reshape(Dd, Du * m)
        dn = torch.sparse.mm(Td, dn).reshape(Dd, Du, m).permute(1, 0, 2).reshape(Du * Dd, m)
        return up + dn + diag * x

    return H


def _complex_apply(H, x):
    """H x for one complex vector."""
    y = H(torch.stack([x.real, x.imag], dim=1))
    return torch.complex(y[:, 0], y[:, 1])


def _cocg(apply, b, shifts, tol, maxit):
    """(A - s_k) x_k = b for every shift by shifted conjugate-orthogonal conjugate gradients."""
    ns = len(shifts)
    s = torch.tensor(shifts, dtype=torch.complex128, device="cuda")
    x = torch.zeros((ns, b.numel()), dtype=torch.complex128, device="cuda")
    pk = torch.zeros_like(x)
    r, p = b.clone(), torch.zeros_like(b)
    z, zp = torch.ones_like(s), torch.ones_like(s)
    bn = float(torch.linalg.vector_norm(b))
    rho, al, be = torch.sum(r * r), torch.ones((), dtype=torch.complex128, device="cuda"), torch.zeros((), dtype=torch.complex128, device="cuda")
    live = torch.ones(ns, dtype=torch.bool, device="cuda")
    for it in range(maxit):
        p = r + be * p
        v = apply(p)
        a = rho / torch.sum(p * v)
        zn = (1 - a * s) * z + (a * be / al) * (z - zp)
        on = live.to(torch.complex128)                     # a finished shift keeps x and p
        f, g, h = torch.where(live, (zp / z) ** 2 * be, on + 1), on / z, on * (z / zn * a)
        pk.mul_(f[:, None]).addcmul_(g[:, None], r[None, :])
        x.addcmul_(pk, h[:, None])
        r = r - a * v
        z, zp = torch.where(live, zn, z), torch.where(live, z, zp)
        new = torch.sum(r * r)
        be, rho, al = new / rho, new, a
        live = live & (torch.linalg.vector_norm(r) / z.abs() > tol * bn)
        if it % 8 == 7:
            if not bool(live.any()):
                break
            t = float(torch.linalg.vector_norm(r)) / bn    # the seed residual falls first: keep r, p and zeta in range
            if t < 1e-20:
                u = 2.0 ** -round(math.log2(t))
                r, p, z, zp, rho = r * u, p * u, z * u, zp * u, rho * (u * u)
    return x


def _fraction(H, phi, E0, w, depth):
    """-(1/pi) Im <phi|(E0 + w + i eta - H)^{-1}|phi> by a Lanczos fraction of fixed depth."""
    n0 = float(torch.sum(phi.abs() ** 2))
    q, qp, a, b = phi / math.sqrt(n0), torch.zeros_like(phi), [], [0.0]
    for _ in range(depth):
        y = _complex_apply(H, q) - b[-1] * qp
        a.append(float(torch.sum((q.conj() * y).real)))
        y = y - a[-1] * q
        b.append(float(torch.linalg.vector_norm(y)))
        qp, q = q, y / b[-1]
    z = E0 + w + 1j * ETA
    f = np.zeros_like(z)
    for j in range(depth - 1, -1, -1):
        f = 1.0 / (z - a[j] - (b[j + 1] ** 2 if j + 1 < depth else 0.0) * f)
    return -(n0 * f).imag / np.pi


def _dense(H, D):
    out = torch.empty((D, D), dtype=torch.float64, device="cuda")
    for i in range(0, D, 512):
        m = min(512, D - i)
        e = torch.zeros((D, m), dtype=torch.float64, device="cuda")
        e[torch.arange(i, i + m), torch.arange(m)] = 1.0
        out[:, i:i + m] = H(e)
    return 0.5 * (out + out.T)


def _lehmann(c, u, uc, w_in, w):
    """The map from full diagonalisation of H and H' (core site 0, up channel), and E_G."""
    L, nu, nd = c["L"], c["nu"], c["nd"]
    E, V = torch.linalg.eigh(_dense(_hamiltonian(c, False, u, uc), _dim(L, nu, nd)))
    ci = dict(c, nu=nu + 1)
    Ep, Vp = torch.linalg.eigh(_dense(_hamiltonian(ci, True, u, uc), _dim(L, nu + 1, nd)))
    il, ih = _created(L, nu)
    lo, hi = math.comb(L, nu), math.comb(L, nu + 1)
    Dd = math.comb(L, nd)
    G = V[:, 0].reshape(lo, Dd)
    b = torch.zeros((hi, Dd), dtype=torch.float64, device="cuda")
    b[ih] = G[il]
    cb = Vp.T @ b.reshape(-1)
    out = np.zeros((len(w_in), len(w)))
    for k, wi in enumerate(w_in):
        d = Ep - E[0] - wi
        coef = torch.stack([cb * d, cb * GAMMA], dim=1) / (d * d + GAMMA * GAMMA)[:, None]
        psi = (Vp @ coef).reshape(hi, Dd, 2)
        phi = torch.zeros((lo, Dd, 2), dtype=torch.float64, device="cuda")
        phi[il] = psi[ih]
        wt = ((V.T @ phi.reshape(-1, 2)) ** 2).sum(dim=1)
        x = (E - E[0])[:, None] - torch.tensor(w, device="cuda")[None, :]
        out[k] = ((wt[:, None] * ETA / (x * x + ETA * ETA)).sum(dim=0) / math.pi).cpu().numpy()
    return out, float(E[0])


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    wide = dict(c, mixed=False)
    if kind == "apply":
        H = _hamiltonian(c, c["core"])
        x = _vectors(c, seed, c["nvec"], _dim(c["L"], c["nu"], c["nd"])).to(torch.complex128)
        return torch.stack([_complex_apply(H, v) + complex(0.33 * c["L"], -GAMMA) * v for v in x])
    if kind in ("solve", "csr"):
        if kind == "solve":
            H = _hamiltonian(c, True, *_couplings(c, seed))
            b, E = _rhs(c, seed)
            b = b.to(torch.complex128)
            c0, shifts = _solve_system(c, E)
            apply = lambda v: _complex_apply(H, v) + c0 * v  # noqa: E731
        else:
            rowptr, col, val = _csr(c, seed)
            A = torch.sparse_csr_tensor(torch.tensor(rowptr), torch.tensor(col.astype(np.int64)), torch.tensor(val),
                                        (c["n"], c["n"]), device="cuda")
            s0, shifts = _csr_shifts(c, seed)
            b = _vectors(c, seed, 1, c["n"])[0].to(torch.complex128)
            apply = lambda v: _complex_apply(lambda m: A @ m, v) - s0 * v  # noqa: E731
        return {"x": _cocg(apply, b, shifts, 1e-9 if c["mixed"] else 1e-13, 3000), "converged": None}
    if kind == "cf":
        H = _hamiltonian(c, False)
        phi = _vectors(c, seed, c["nvec"], _dim(c["L"], c["nu"], c["nd"])).to(torch.complex128)
        w = _grids(c)[1]
        return {"I": np.stack([_fraction(H, v, E_SITE * c["L"], w, c["depth"]) for v in phi]), "depth": None}
    if kind == "map" and _dim(c["L"], c["nu"], c["nd"]) <= 5000 and c["nu"] < c["L"]:
        u, uc = _couplings(c, seed)
        I, E = _lehmann(wide, u, uc, *_grids(c))
        return {"I": I, "E": E}
    if kind == "ground" and _dim(c["L"], c["nu"], c["nd"]) <= 5000:
        u, uc = _couplings(c, seed)
        E = torch.linalg.eigvalsh(_dense(_hamiltonian(c, False, u, uc), _dim(c["L"], c["nu"], c["nd"])))
        return {"E": float(E[0]), "g": None}
    return None
