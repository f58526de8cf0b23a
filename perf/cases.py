"""What a user has this library do, as cases that can be timed.

Every case is one pass through the public binding (`paper_1004_3354_gb300`): a
Hamiltonian-vector product, an eigensolve, a batch of sectors, or a Green's
function, on the model families of the repository: the Anderson impurity
(Eq. 2), the three-orbital Kanamori impurity (Sec. 4) and the Hubbard ring
(Eq. 1).  Model parameters, start vectors and states come from the seed.

Keys of a case:
  op      "hv" (ed_apply_h), "lanczos" (full reorthogonalisation), "lanczos3"
          (three-vector), "trlan" (thick restart), "batch" (all sectors of a
          model), "greens" (continued fraction)
  family  "aim", "kanamori", "hubbard"
  n_s, n_up, n_dn   sites and particles (n_s alone for "batch")
  prec    "fp64", "df64", "fp32"
  k       lowest states wanted (eigensolves);  depth, n_w, z  (greens)
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1004_3354_gb300 as ed
import workloads as W

TOL = 1e-10      # residual tolerance of the eigensolves, as in the repository's benchmark
BETA = 40.0      # inverse temperature of the Green's function


def listed():
    return [
        # One H*v of the smallest impurity the tests and smoke() use (dim 400): a
        # call is launch latency, as in every step of a small DMFT solve.
        dict(name="hv_aim6_fp64", op="hv", family="aim", n_s=6, n_up=3, n_dn=3, prec="fp64"),
        # H*v of the N_s = 12 impurity (dim 853,776), the ordinary size of a served
        # request and the largest sector of the 169-sector batch.
        dict(name="hv_kan12_df64", op="hv", family="kanamori", n_s=12, n_up=6, n_dn=6, prec="df64"),
        # The benchmark's headline: H*v at N_s = 15, sector (7, 8), dim 41,409,225,
        # in the production double-float format, ...
        dict(name="hv_kan15_df64", op="hv", family="kanamori", n_s=15, n_up=7, n_dn=8, prec="df64"),
        # ... with float vectors (the served format) ...
        dict(name="hv_kan15_fp32", op="hv", family="kanamori", n_s=15, n_up=7, n_dn=8, prec="fp32"),
        # ... and with plain FP64 vectors (the default format of the binding).
        dict(name="hv_kan15_fp64", op="hv", family="kanamori", n_s=15, n_up=7, n_dn=8, prec="fp64"),
        # H*v of the largest sector that is served (N_s = 16, dim 165,636,900).
        dict(name="hv_kan16_fp32", op="hv", family="kanamori", n_s=16, n_up=8, n_dn=8, prec="fp32"),
        # H*v of the Hubbard cluster (Eq. 1) with U on every site: the general
        # kernels, at the (7, 7) sector of 14 sites, dim 11,778,624.
        dict(name="hv_hub14_df64", op="hv", family="hubbard", n_s=14, n_up=7, n_dn=7, prec="df64"),
        # The lowest states of one sector with full reorthogonalisation.
        dict(name="lanczos_kan12_df64", op="lanczos", family="kanamori", n_s=12, n_up=6, n_dn=6, prec="df64", k=4),
        # Ground state of a DMFT impurity (one orbital, a ragged sector) by the
        # three-vector recurrence with the second pass for its vector.
        dict(name="lanczos3_aim13_fp64", op="lanczos3", family="aim", n_s=13, n_up=7, n_dn=6, prec="fp64", k=1),
        # A served impurity solve's eigensolve: the four lowest states by thick restart.
        dict(name="trlan_kan13_df64", op="trlan", family="kanamori", n_s=13, n_up=7, n_dn=6, prec="df64", k=4),
        # All 121 sectors of a ten-site impurity together (the sum of Eq. 3 runs
        # over every sector): 1,048,576 states from dimension 1 to 63,504.
        dict(name="batch_kan10_fp64", op="batch", family="kanamori", n_s=10, prec="fp64", k=8),
        # G(i w_n) of an impurity orbital from its ground state, 1024 Matsubara
        # points: one solve per DMFT iteration.
        dict(name="greens_kan12_df64", op="greens", family="kanamori", n_s=12, n_up=6, n_dn=6, prec="df64",
             depth=100, n_w=1024),
    ]


def draw(rng):
    """One more case of the ranges above: H*v over three decades and more of
    sector dimension in every format and family, and solves up to the listed ones'
    size."""
    op = rng.choice(["hv", "hv", "hv", "hv", "lanczos", "lanczos3", "trlan", "batch", "greens"])
    if op == "batch":
        return dict(op=op, family="kanamori", n_s=rng.randint(7, 10), prec=rng.choice(["fp64", "df64"]),
                    k=rng.randint(1, 8))
    family = rng.choice(["kanamori", "kanamori", "aim", "hubbard"] if op == "hv" else ["kanamori", "aim"])
    lo, hi = {"hv": (6, 15), "lanczos": (8, 12)}.get(op, (8, 13))
    n_s = rng.randint(lo, hi)
    half = n_s // 2
    n_up = max(1, half + rng.choice([-2, -1, 0, 0, 1]))
    n_dn = max(1, half + rng.choice([-1, 0, 0, 1, 2]))
    c = dict(op=op, family=family, n_s=n_s, n_up=n_up, n_dn=n_dn,
             prec=rng.choice(["fp64", "df64", "fp32"] if op == "hv" else ["fp64", "df64"]))
    if op == "hv":
        return c
    if op == "greens":
        return dict(c, depth=rng.randint(20, 100), n_w=int(2 ** rng.uniform(6, 10.5)))
    return dict(c, k=1 if op == "lanczos3" else rng.randint(1, 4))


# ------------------------------------------------------------------- inputs
def _model(case, seed):
    s = int(seed) % (1 << 31)
    if case["family"] == "aim":
        return W.aim(case["n_s"], seed=s)
    if case["family"] == "kanamori":
        return W.kanamori(case["n_s"], seed=s)
    r = np.random.default_rng(s)
    return W.hubbard_cluster(case["n_s"], t=1.0, U=float(r.uniform(2.0, 8.0)), tp=float(r.uniform(0.0, 0.3)))


def _dims(case):
    return math.comb(case["n_s"], case["n_up"]), math.comb(case["n_s"], case["n_dn"])


def _randn(n, seed, device):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed) + 77)
    return torch.randn(n, generator=g, dtype=torch.float64, device=device)


def _store(x, prec):
    """FP64 vector in a storage format: as it is, float, or {hi, lo} float pairs."""
    if prec == "fp64":
        return x
    hi = x.float()
    if prec == "fp32":
        return hi
    return torch.stack([hi, (x - hi.double()).float()], dim=1).reshape(-1)


class _State:
    """What the program keeps: a context and what it made in it."""

    def __init__(self):
        self.ctx = ed.ed_ctx_create(torch.cuda.current_device())
        self.sec = self.batch = None

    def __del__(self):
        try:
            if self.sec is not None:
                ed.ed_sector_destroy(self.sec)
            if self.batch is not None:
                ed.ed_batch_destroy(self.batch)
            ed.ed_ctx_destroy(self.ctx)
        except Exception:
            pass


def _sectors(n_s):
    return [(a, b) for a in range(n_s + 1) for b in range(n_s + 1)]


def prepare(case, seed):
    st = _State()
    st.case = case
    st.model = ed.Model(_model(case, seed))
    st.seed = int(seed) % (1 << 31) + 1
    op, prec = case["op"], case["prec"]
    if op == "batch":
        st.sectors = _sectors(case["n_s"])
        st.batch = ed.ed_batch_create(st.ctx, st.model, st.sectors, prec)
        return st
    du, dd = _dims(case)
    dim = du * dd
    if op == "greens":
        # the ground state that a solve before it has left on the device
        E, psi = _ground(_model(case, seed), case["n_up"], case["n_dn"], seed)
        st.states = [(case["n_up"], case["n_dn"], E, _store(psi, prec))]
        return st
    st.sec = ed.ed_sector_create(st.ctx, st.model, case["n_up"], case["n_dn"], prec)
    if op == "hv":
        st.x = _store(_randn(dim, seed, "cuda"), prec)
        st.y = torch.empty_like(st.x)
    else:
        st.k = min(case["k"], dim)
        st.psi = torch.empty(st.k * dim * ed.elems_per_value(prec), dtype=ed.torch_dtype(prec), device="cuda")
    return st


def run(st):
    c = st.case
    op = c["op"]
    if op == "hv":
        ed.ed_apply_h(st.sec, st.x, st.y)
        return st.y
    if op == "lanczos":
        ev, _, _ = ed.ed_lanczos(st.sec, k=st.k, tol=TOL, max_iter=500, check_every=10, seed=st.seed, evecs=st.psi)
        return ev, st.psi
    if op == "lanczos3":
        ev, _, _ = ed.ed_lanczos(st.sec, k=st.k, tol=TOL, max_iter=500, check_every=10, seed=st.seed, reorth=False,
                                 evecs=st.psi)
        return ev, st.psi
    if op == "trlan":
        ev, _, _ = ed.ed_lanczos_tr(st.sec, k=st.k, tol=TOL, max_basis=40, max_iter=3000, check_every=5, seed=st.seed,
                                    evecs=st.psi)
        return ev, st.psi
    if op == "batch":
        ev, _, _, _ = ed.ed_batch_lanczos(st.batch, len(st.sectors), k=c["k"], tol=TOL, max_iter=500, check_every=10,
                                          seed=st.seed)
        return ev
    return ed.ed_greens_cf(st.ctx, st.model, c["prec"], st.states, BETA, c["n_w"], orbital=st.model.src.orb0,
                           depth=c["depth"])


# --------------------------------------------------------------------- work
def _macs_per_element(case, n_up, n_dn):
    """Mean entries of a row of H: the diagonal, each spin's one-body hops and
    the spin-flip / pair-hop moves (a move i -> j exists in C(n_s-2, n-1) of the
    C(n_s, n) strings)."""
    n_s = case["n_s"]

    def frac(n):
        return n * (n_s - n) / (n_s * (n_s - 1)) if n_s > 1 else 0.0
    bonds = {"aim": n_s - 1, "kanamori": n_s - 3, "hubbard": 2 * n_s}[case["family"]]
    mix = 12 if case["family"] == "kanamori" else 0   # ordered orbital pairs x (spin flip, pair hop)
    return 1 + 2 * bonds * (frac(n_up) + frac(n_dn)) + mix * frac(n_up) * frac(n_dn)


def work(case):
    """x read once and y written once per H*v; with reorthogonalisation the
    basis read once per pass of the twice-repeated projection.  The numbers of
    steps are those that these models take to converge at TOL."""
    eb = 4 if case["prec"] == "fp32" else 8
    op = case["op"]
    if op == "batch":
        dim = 4 ** case["n_s"]
        mac = _macs_per_element(case, case["n_s"] // 2, case["n_s"] // 2)
        steps = 70 + 20 * case["k"]
    else:
        du, dd = _dims(case)
        dim = du * dd
        mac = _macs_per_element(case, case["n_up"], case["n_dn"])
        steps = {"hv": 1, "lanczos": 80 + 25 * case.get("k", 1), "lanczos3": 2 * 90, "trlan": 80 + 30 * case.get("k", 1),
                 "greens": 2 * case.get("depth", 1)}[op]
        if op != "hv":
            steps = min(steps, 2 * dim)
    hv_b, hv_f = 2.0 * dim * eb, 2.0 * mac * dim
    if op == "hv":
        return {"bytes": hv_b, "flops": hv_f}
    if op in ("lanczos3", "greens"):      # q_{j+1} from H q_j, q_j, q_{j-1}: one more read and write
        return {"bytes": steps * (hv_b + 2.0 * dim * eb), "flops": steps * (hv_f + 10.0 * dim)}
    mean_basis = {"lanczos": steps / 2, "batch": steps / 2, "trlan": 25}[op]
    return {"bytes": steps * (hv_b + 2 * mean_basis * dim * eb),
            "flops": steps * (hv_f + 2 * 4 * mean_basis * dim)}


# -------------------------------------------------------- plain 64-bit values
def _strings(n_s, n):
    s = np.arange(1 << n_s, dtype=np.int64)
    pop = np.zeros_like(s)
    for i in range(n_s):
        pop += (s >> i) & 1
    return s[pop == n], pop


class _PlainH:
    """H of a sector on a (D_up, D_dn) float64 array, term by term in torch."""

    def __init__(self, m, n_up, n_dn, device):
        self.m, n_s = m, m.n_s
        T = np.asarray(m.T)
        orbs = [m.orb0 + a for a in range(m.n_orb)]
        spins = []
        for n in (n_up, n_dn):
            s, pop = _strings(n_s, n)
            rank = np.zeros(1 << n_s, dtype=np.int64)
            rank[s] = np.arange(len(s))

            def move(i, j):
                """c+_i c_j: rows (i occupied, j empty in the row string), sources, signs."""
                rows = np.nonzero(((s >> i) & 1 == 1) & ((s >> j) & 1 == 0))[0]
                between = ((1 << max(i, j)) - 1) & ~((1 << (min(i, j) + 1)) - 1)
                sign = 1.0 - 2.0 * (pop[s[rows] & between] & 1)
                src = rank[s[rows] ^ (1 << i) ^ (1 << j)]
                return rows, src, sign
            hops = [[], [], []]
            for i in range(n_s):
                for j in range(n_s):
                    if i != j and T[i, j] != 0.0:
                        r, c, v = move(i, j)
                        hops[0].append(r)
                        hops[1].append(c)
                        hops[2].append(T[i, j] * v)
            cat = [np.concatenate(h) if h else np.zeros(0) for h in hops]
            D = len(s)
            hop = torch.sparse_coo_tensor(torch.from_numpy(np.stack([cat[0], cat[1]]).astype(np.int64)),
                                          torch.from_numpy(cat[2].astype(np.float64)), (D, D)).to(device).coalesce()
            occ = np.stack([(s >> i) & 1 for i in range(n_s)], axis=1).astype(np.float64)
            e = occ @ np.diag(T)
            for a in range(m.n_orb):
                for b in range(a + 1, m.n_orb):
                    e = e + (m.Up - m.J) * occ[:, orbs[a]] * occ[:, orbs[b]]
            moves = {(a, b): move(a, b) for a in orbs for b in orbs if a != b}
            spins.append(dict(hop=hop.to_sparse_csr(), e=torch.from_numpy(e).to(device),
                              occ=torch.from_numpy(occ).to(device),
                              moves={q: tuple(torch.from_numpy(v).to(device) for v in mv) for q, mv in moves.items()}))
        self.up, self.dn = spins
        V = np.diag(np.asarray(m.U_site, dtype=np.float64))
        for a in orbs:
            for b in orbs:
                if a != b:
                    V[a, b] += m.Up
        self.diag = self.up["e"][:, None] + self.dn["e"][None, :] + self.up["occ"] @ torch.from_numpy(V).to(device) @ self.dn["occ"].T

    def __call__(self, X):
        Y = self.diag * X
        Y += self.up["hop"] @ X
        Y += (self.dn["hop"] @ X.T.contiguous()).T
        m = self.m
        for (a, b), (ru, cu, su) in self.up["moves"].items():
            for J, q in ((m.Jsf, (b, a)), (m.Jph, (a, b))):
                if J == 0.0:
                    continue
                rd, cd, sd = self.dn["moves"][q]
                if ru.numel() and rd.numel():
                    Y[ru[:, None], rd[None, :]] += J * su[:, None] * sd[None, :] * X[cu[:, None], cd[None, :]]
        return Y


def _lowest(H, shape, k, seed, steps, want_vec=False):
    """Lowest k values (and the lowest vector) by plain Lanczos, every vector
    kept and every new one orthogonalised twice."""
    dev = H.diag.device
    dim = shape[0] * shape[1]
    steps = min(steps, dim)
    v = _randn(dim, seed + 5, dev)
    V = torch.empty(steps, dim, dtype=torch.float64, device=dev)
    a, b = torch.zeros(steps, dtype=torch.float64, device=dev), torch.zeros(steps, dtype=torch.float64, device=dev)
    V[0] = v / v.norm()
    m = steps
    for j in range(steps):
        w = H(V[j].view(shape)).reshape(-1)
        a[j] = V[j] @ w
        for _ in range(2):
            w -= V[: j + 1].T @ (V[: j + 1] @ w)
        b[j] = w.norm()
        if j + 1 < steps:
            V[j + 1] = w / b[j]
        if j % 10 == 9 and float(b[j]) < 1e-10:
            m = j + 1
            break
    Tm = torch.diag(a[:m]) + torch.diag(b[: m - 1], 1) + torch.diag(b[: m - 1], -1)
    w, S = torch.linalg.eigh(Tm)
    return w[:k], (S[:, 0] @ V[:m]) if want_vec else None


_GROUND = {}


def _ground(m, n_up, n_dn, seed):
    """Energy and vector of the sector's ground state, from plain torch."""
    key = (m.name, repr(sorted(m.params.items(), key=str)), n_up, n_dn, int(seed))
    if key not in _GROUND:
        H = _PlainH(m, n_up, n_dn, "cuda")
        w, v = _lowest(H, tuple(H.diag.shape), 1, seed, 100, want_vec=True)
        if len(_GROUND) > 3:
            _GROUND.clear()
        _GROUND[key] = (float(w[0]), v / v.norm())
    return _GROUND[key]


def exact(case, seed):
    op, prec = case["op"], case["prec"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    m = _model(case, seed)
    if op == "batch":
        if case["n_s"] > 8:
            return None       # a full diagonalisation of every sector: too long
        out = torch.full((len(_sectors(case["n_s"])), case["k"]), float("nan"), dtype=torch.float64)
        for i, (nu, nd) in enumerate(_sectors(case["n_s"])):
            H = _PlainH(m, nu, nd, dev)
            shape = tuple(H.diag.shape)
            w, _ = _lowest(H, shape, case["k"], 3, 160)
            out[i, : len(w)] = w.cpu()
        return out
    H = _PlainH(m, case["n_up"], case["n_dn"], dev)
    shape = tuple(H.diag.shape)
    dim = shape[0] * shape[1]
    if op == "hv":
        x = _store(_randn(dim, seed, dev), prec)
        x = x.double() if prec != "df64" else x.double().view(-1, 2).sum(1)
        y = H(x.view(shape)).reshape(-1)
        return _store(y, "df64") if prec == "df64" else y
    if op in ("lanczos", "trlan", "lanczos3"):
        k = min(case["k"], dim)
        w, _ = _lowest(H, shape, k, seed, 150 if k == 1 else 300)
        return w, None        # the vectors' signs are the solver's own
    return None               # a depth-L continued fraction in exact arithmetic is not what L rounded steps give
