"""Performance cases of libed: what users of the solver have it do, through its public calls.

Kinds of case:
  hpsi     one product y = H x on device vectors (ed_hpsi), the step every Krylov method repeats
  ground   one ground state with its vector (ed_cluster_create, ed_ground_state, ed_ground_vector)
  solve    one impurity solve: ground state and Green function of a cluster, create to destroy
  batch    many small clusters in one call (ed_batch_solve)
  lattice  the lattice steps that consume G: periodized CPT, CDMFT target, distance and gradient
  sym      a solve in one irrep of the cluster's mirror group (ed_sym_*)

G of runs with FP32 vectors is handed on as complex64: it carries single precision.
"""

import itertools
import math

import numpy as np
import torch

from paper_2305_18643_gb300 import ed
from paper_2305_18643_gb300 import workloads as W

BETA = 50.0  # inverse temperature of the Matsubara grids
ETA = 0.05   # broadening on the real axis


# ------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest product: plain 2x4 cluster, 4,900 states, where launch latency counts
        dict(name="hpsi_2x4_f64", kind="hpsi", cluster="ladder", size=4, n_up=4, n_dn=4, fp32=False, pad=False),
        # a CDMFT impurity (2x2 plaquette + 8 bath orbitals), 853,776 states, contiguous rows
        dict(name="hpsi_impurity12_f64", kind="hpsi", cluster="impurity", size=8, n_up=6, n_dn=6, fp32=False, pad=False),
        # a Green-function sector of the 14-orbital ladder: unequal, odd dimensions, FP32 vectors
        dict(name="hpsi_2x7_f32", kind="hpsi", cluster="ladder", size=7, n_up=8, n_dn=7, fp32=True, pad=True),
        # the N+1 sector of the 4x4 cluster (147 M states): the product of its band Lanczos
        dict(name="hpsi_4x4_f32", kind="hpsi", cluster="4x4", size=4, n_up=9, n_dn=8, fp32=True, pad=True),
        # the same cluster's ground-state sector (166 M states) in the default precision
        dict(name="hpsi_4x4_f64", kind="hpsi", cluster="4x4", size=4, n_up=8, n_dn=8, fp32=False, pad=True),
        # the plain solve: 2x4 cluster, continued fractions on 1000 real frequencies
        dict(name="solve_2x4_f64", kind="solve", cluster="ladder", size=4, fp32=False, band=False, matsubara=False,
             n_freq=1000),
        # one iteration of a CDMFT loop: impurity solve on Matsubara frequencies, band Lanczos
        dict(name="solve_impurity12_f64", kind="solve", cluster="impurity", size=8, fp32=False, band=True,
             matsubara=True, n_freq=1000),
        # a served 14-orbital request with FP32 vectors and the FP64 refinement of its ground state
        dict(name="solve_2x7_f32", kind="solve", cluster="ladder", size=7, fp32=True, band=True, matsubara=True,
             n_freq=2048),
        # the largest: ground state of the 4x4 periodic cluster, FP32 vectors refined to FP64
        dict(name="ground_4x4_f32", kind="ground", cluster="4x4", size=4, n_up=8, n_dn=8, fp32=True),
        # a sweep over many small clusters of different size and filling in one call
        dict(name="batch_64_f64", kind="batch", n=64, max_orb=7, fp32=False, matsubara=False, n_freq=512),
        # the lattice half of a CDMFT iteration on the square lattice tiled by 2x2 plaquettes
        dict(name="lattice_2x2", kind="lattice", width=2, height=2, n_bath=8, k_cpt=64, k_cdmft=16, n_freq=256,
             n_cand=64),
        # a symmetric cluster solved in the fully symmetric irrep of its two mirrors
        dict(name="sym_3x4_f64", kind="sym", width=4, height=3, n_freq=64),
    ]


def draw(rng):
    """One more case of the ranges above."""
    kind = rng.choice(["hpsi", "hpsi", "hpsi", "solve", "solve", "ground", "batch", "lattice", "sym"])
    if kind in ("hpsi", "ground"):
        cluster = rng.choice(["ladder", "chain", "impurity", "4x4"])
        size = {"ladder": rng.randint(3, 7), "chain": rng.randint(6, 14), "impurity": rng.randint(2, 9), "4x4": 4}[cluster]
        n = orbitals(cluster, size)
        if kind == "ground":
            fp32 = rng.random() < 0.5
            n_up = rng.randint(5, 7 if fp32 else 5) if cluster == "4x4" else n // 2
            return dict(kind=kind, cluster=cluster, size=size, n_up=n_up, n_dn=n_up if cluster == "4x4" else n - n_up,
                        fp32=fp32)
        return dict(kind=kind, cluster=cluster, size=size, n_up=rng.randint(max(2, n // 2 - 2), n // 2 + 1),
                    n_dn=rng.randint(max(2, n // 2 - 2), n // 2 + 1), fp32=rng.random() < 0.5, pad=rng.random() < 0.5)
    if kind == "solve":
        cluster = rng.choice(["ladder", "impurity"])
        matsubara = rng.random() < 0.7
        big = 6 if matsubara else 4
        size = rng.randint(3, big) if cluster == "ladder" else 2 * rng.randint(1, big - 2)
        # FP32 vectors on the real axis amplify their rounding near poles: single precision solves go
        # with the Matsubara axis
        return dict(kind=kind, cluster=cluster, size=size, fp32=matsubara and rng.random() < 0.4,
                    band=matsubara and rng.random() < 0.6, matsubara=matsubara,
                    n_freq=int(round(math.exp(rng.uniform(math.log(100), math.log(2048))))))
    if kind == "batch":
        matsubara = rng.random() < 0.5
        return dict(kind=kind, n=int(round(math.exp(rng.uniform(math.log(4), math.log(64))))),
                    max_orb=rng.randint(5, 8 if matsubara else 7), fp32=False, matsubara=matsubara,
                    n_freq=rng.randint(64, 512))
    if kind == "lattice":
        w, h = rng.choice([(2, 1), (2, 2), (3, 1), (3, 2), (4, 2)])
        return dict(kind=kind, width=w, height=h, n_bath=rng.randint(2, 10), k_cpt=rng.randint(16, 40),
                    k_cdmft=rng.randint(8, 16), n_freq=rng.randint(32, 200), n_cand=rng.randint(1, 64))
    w, h = rng.choice([(3, 2), (4, 2), (5, 2), (6, 2), (3, 3), (4, 3)])
    return dict(kind=kind, width=w, height=h, n_freq=rng.randint(32, 256))


def orbitals(cluster, size):
    return {"ladder": 2 * size, "chain": size, "impurity": 4 + size, "4x4": 16}[cluster]


def make_cluster(cluster, size, n_up, n_dn, seed):
    """A cluster of the given shape whose couplings follow from the seed."""
    rng = np.random.default_rng(seed)
    if cluster == "4x4":
        c = W.periodic_4x4()
    elif cluster == "impurity":
        theta = np.zeros((4, size))
        theta[np.arange(size) % 4, np.arange(size)] = rng.uniform(0.2, 0.8, size)
        c = dict(t=W.lattice_hopping(2, 2, tp=0.3), eps=rng.uniform(-2.0, 2.0, size), theta=theta)
    else:
        H = 2 if cluster == "ladder" else 1
        tp = 0.3 if H == 2 and size > 4 else 0.0
        t = W.lattice_hopping(size, H, tp=tp, rng=np.random.default_rng(size), seeded_tp_sign=True)
        c = dict(t=t, eps=np.zeros(0), theta=np.zeros((t.shape[0], 0)))
    U = (4.0 if cluster == "ladder" and size <= 4 else 8.0) + rng.uniform(-0.5, 0.5)
    return dict(c, U=np.full(c["t"].shape[0], U), mu=U / 2, n_up=n_up, n_dn=n_dn)


def solve_cluster(case, seed):
    n = orbitals(case["cluster"], case["size"])
    return make_cluster(case["cluster"], case["size"], n // 2, n - n // 2, seed)


def grid(case):
    return W.matsubara_grid(case["n_freq"], BETA) if case.get("matsubara", True) else W.real_grid(case["n_freq"])


def batch_clusters(case, seed):
    """The seeded family of small clusters, its couplings scaled by factors that follow from the seed."""
    rng = np.random.default_rng(seed)
    family = []
    for c in W.batched_family(case["n"], max_orb=case["max_orb"]):
        U = c["U"] * rng.uniform(0.9, 1.1)
        family.append(dict(c, t=c["t"] * rng.uniform(0.9, 1.1), U=U, mu=float(U[0]) / 2))
    return family


def by_sites(G):
    """The clusters' Green functions [2, n_freq, ns, ns], one array per number of sites ns."""
    return {str(ns): np.stack([g for g in G if g.shape[-1] == ns]) for ns in sorted({g.shape[-1] for g in G})}


def lattice_inputs(case, seed):
    """Superlattice, a cluster Green function in Lehmann form, its bath and trial baths."""
    rng = np.random.default_rng(seed)
    L, nb = case["width"] * case["height"], case["n_bath"]
    lat = W.square_superlattice(case["width"], case["height"], -1.0, 0.3 if case["height"] > 1 else 0.0)
    z = 1j * W.matsubara_grid(case["n_freq"], BETA)
    q, _ = np.linalg.qr(rng.standard_normal((6 * L, L)))
    poles = rng.uniform(-6.0, 6.0, 6 * L)
    Gc = np.einsum("ra,zr,rb->zab", q, 1.0 / (z[:, None] - poles[None, :]), q)
    theta, eps = rng.uniform(0.1, 0.8, (L, nb)), rng.uniform(-2.0, 2.0, nb)
    Gamma = np.einsum("ia,za,ja->zij", theta, 1.0 / (z[:, None] - eps[None, :]), theta)
    dim = np.asarray(lat["E"]).shape[0]
    trial = (theta + 0.1 * rng.standard_normal((case["n_cand"], L, nb)), eps + 0.1 * rng.standard_normal((case["n_cand"], nb)))
    w = 1.0 / np.abs(z)
    return dict(lat=lat, z=z, Gc=Gc, Gamma=Gamma, trial=trial, weights=w / w.sum(),
                k_cpt=W.reduced_zone(np.eye(dim), [case["k_cpt"]] * dim),
                k_cdmft=W.reduced_zone(lat["E"], [case["k_cdmft"]] * dim))


def sym_cluster(case, seed):
    w, h = case["width"], case["height"]
    n = w * h
    U = 4.0 + np.random.default_rng(seed).uniform(-0.5, 0.5)
    c = dict(t=W.lattice_hopping(w, h), U=np.full(n, U), mu=U / 2, eps=np.zeros(0), theta=np.zeros((n, 0)),
             n_up=n // 2, n_dn=n // 2)
    mirrors = [[(w - 1 - s % w) + w * (s // w) for s in range(n)], [s % w + w * (h - 1 - s // w) for s in range(n)]]
    return c, mirrors


# ------------------------------------------------------------------------------------------ prepare, run
def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case)
    if kind == "hpsi":
        c = make_cluster(case["cluster"], case["size"], case["n_up"], case["n_dn"], seed)
        state["cl"] = ed.Cluster(c)
        du, dd = ed.ed_sector_dims(state["cl"].h, case["n_up"], case["n_dn"])
        x = hpsi_vector(case, seed, du, dd)
        state.update(x=x, y=torch.zeros_like(x), dd=dd)
    elif kind in ("solve", "ground"):
        state["c"] = (solve_cluster(case, seed) if kind == "solve" else
                      make_cluster(case["cluster"], case["size"], case["n_up"], case["n_dn"], seed))
        if kind == "solve":
            state["omega"] = grid(case)
        else:
            n = orbitals(case["cluster"], case["size"])
            state["v"] = torch.empty((math.comb(n, case["n_up"]), math.comb(n, case["n_dn"])), dtype=torch.float64,
                                     device="cuda")
    elif kind == "batch":
        state.update(clusters=batch_clusters(case, seed), omega=grid(case))
    elif kind == "lattice":
        state.update(lattice_inputs(case, seed))
    else:
        c, mirrors = sym_cluster(case, seed)
        state.update(c=c, mirrors=mirrors, omega=grid(case))
    return state


def hpsi_vector(case, seed, du, dd):
    """A normalized vector of du rows; padded rows (a multiple of 128 elements) hold zeros past dd."""
    ld = (dd + 127) // 128 * 128 if case["pad"] else dd
    g = torch.Generator("cuda").manual_seed(seed)
    x = torch.zeros((du, ld), dtype=torch.float32 if case["fp32"] else torch.float64, device="cuda")
    x[:, :dd] = torch.randn((du, dd), dtype=torch.float32, device="cuda", generator=g)
    x[:, :dd] /= torch.linalg.vector_norm(x)
    return x


def run(state):
    case = state["case"]
    kind = case["kind"]
    fp32 = bool(case.get("fp32"))
    precision = ed.ED_FP32 if fp32 else ed.ED_FP64
    if kind == "hpsi":
        x, y = state["x"], state["y"]
        ed.ed_hpsi(state["cl"].h, case["n_up"], case["n_dn"], precision, x.data_ptr(), y.data_ptr(), x.shape[1],
                   torch.cuda.current_stream().cuda_stream)
        return y[:, :state["dd"]]
    if kind == "ground":
        with ed.Cluster(state["c"], precision=precision, seed=1234) as cl:
            _, E0, _, _ = cl.ground_state()
            ed.ed_ground_vector(cl.h, case["n_up"], case["n_dn"], state["v"].data_ptr())
        return dict(E0=E0, vector=state["v"])
    if kind == "solve":
        with ed.Cluster(state["c"], precision=precision, gf_method=ed.ED_GF_BAND if case["band"] else ed.ED_GF_CF,
                        seed=1234) as cl:
            _, E0, _, _ = cl.ground_state()
            G = cl.green(state["omega"], ETA, ed.ED_AXIS_MATSUBARA if case["matsubara"] else ed.ED_AXIS_REAL)
        return dict(E0=E0, G=G.astype(np.complex64) if fp32 else G)
    if kind == "batch":
        E0, _, _, _, G = ed.ed_batch_solve(state["clusters"], precision=precision, omega=state["omega"], eta=ETA,
                                           axis=ed.ED_AXIS_MATSUBARA if case["matsubara"] else ed.ED_AXIS_REAL, seed=7)
        return dict(E0=E0, G=by_sites(G))
    if kind == "lattice":
        s = state
        G = ed.ed_cpt_green(s["lat"], s["Gc"], s["k_cpt"], ed.ED_CPT_PERIODIZED, Gamma=s["Gamma"])
        A = ed.ed_cdmft_target(s["lat"], s["Gc"], s["k_cdmft"], Gamma=s["Gamma"])
        d, grad = ed.ed_cdmft_distance(s["trial"][0], s["trial"][1], s["z"], s["weights"], A, grad=True)
        return dict(G=G, A=A, d=d, grad=grad)
    n = case["width"] * case["height"]
    with ed.Cluster(state["c"], seed=1234) as cl:
        sym = ed.ed_sym_create(cl.h, state["mirrors"], [1, 1])
        try:
            E0 = ed.ed_sym_ground_state(sym)[0]
            G = ed.ed_sym_green(sym, state["omega"], n, axis=ed.ED_AXIS_MATSUBARA)
        finally:
            ed.ed_sym_destroy(sym)
    return dict(E0=E0, G=G)


# ------------------------------------------------------------------------------------------ work
def hops(c, n):
    """Mean number of hops per state of one spin with n particles."""
    h = one_body(c)
    L = h.shape[0]
    bonds = np.count_nonzero(h) - np.count_nonzero(np.diag(h))
    return bonds * n * (L - n) / (L * (L - 1)) if L > 1 else 0.0


def product_work(c, n_up, n_dn, size, vectors):
    """Bytes and flops of one product that reads and writes `vectors` vectors of the sector."""
    L = one_body(c).shape[0]
    d = math.comb(L, n_up) * math.comb(L, n_dn)
    return vectors * size * d, 2.0 * d * (hops(c, n_up) + hops(c, n_dn) + 1)


def work(case):
    kind = case["kind"]
    size = 4 if case.get("fp32") else 8
    if kind == "hpsi":
        c = make_cluster(case["cluster"], case["size"], case["n_up"], case["n_dn"], 0)
        b, f = product_work(c, case["n_up"], case["n_dn"], size, 2)
        return dict(bytes=b, flops=f)
    # Krylov methods: a step reads two vectors and writes one.  100 steps resolve a ground state; a
    # Green function takes about 50 steps per starting vector on the Matsubara axis, 400 on the real one
    if kind in ("ground", "solve", "sym"):
        if kind == "ground":
            c = make_cluster(case["cluster"], case["size"], case["n_up"], case["n_dn"], 0)
        else:
            c = solve_cluster(case, 0) if kind == "solve" else sym_cluster(case, 0)[0]
        ns, nu, nd = c["t"].shape[0], c["n_up"], c["n_dn"]
        group = 4 if kind == "sym" else 1
        b, f = product_work(c, nu, nd, size, 3)
        b, f = 100 * b / group, 100 * f / group
        if kind != "ground":
            steps = 2 * ns * (50 if case.get("matsubara", True) else 400)
            bg, fg = product_work(c, nu + 1, nd, size, 3)
            b, f = b + steps * bg / group, f + steps * fg / group
        return dict(bytes=b, flops=f)
    if kind == "batch":
        b = f = 0.0
        for c in batch_clusters(case, 0):
            bg, fg = product_work(c, c["n_up"], c["n_dn"], size, 3)
            steps = 100 + 4 * c["t"].shape[0] * (50 if case["matsubara"] else 400)
            b, f = b + steps * bg, f + steps * fg
        return dict(bytes=b, flops=f)
    L, nz = case["width"] * case["height"], case["n_freq"]
    D = 1 if case["height"] == 1 else 2
    points = nz * (case["k_cpt"] ** D + case["k_cdmft"] ** D)
    grad = case["n_cand"] * nz * case["n_bath"] * 24 * L * L
    return dict(bytes=16.0 * nz * (case["k_cpt"] ** D + 3 * L * L), flops=8.0 * points * L ** 3 + grad)


# ------------------------------------------------------------------------------------------ exact, in 64 bits
def one_body(c):
    ns, nb = c["t"].shape[0], len(c["eps"])
    h = np.zeros((ns + nb, ns + nb))
    h[:ns, :ns] = c["t"] - c["mu"] * np.eye(ns)
    h[:ns, ns:] = c["theta"]
    h[ns:, :ns] = c["theta"].T
    h[range(ns, ns + nb), range(ns, ns + nb)] = c["eps"]
    return h


def spin_basis(L, n):
    return np.array(sorted(sum(1 << i for i in s) for s in itertools.combinations(range(L), n)), dtype=np.int64)


def bits(v):
    return np.array([bin(x).count("1") for x in v.tolist()], dtype=np.int64)


class Sector:
    """H of one (n_up, n_dn) sector on vectors psi[u, d], from the bond list of the cluster."""

    def __init__(self, c, n_up, n_dn):
        h = one_body(c)
        L = h.shape[0]
        U = np.zeros(L)
        U[:len(c["U"])] = c["U"]
        self.B = [spin_basis(L, n_up), spin_basis(L, n_dn)]
        occ = [torch.tensor((b[:, None] >> np.arange(L)) & 1, dtype=torch.float64, device="cuda") for b in self.B]
        self.K = [self.hopping(h, b) for b in self.B]
        one = [o @ torch.tensor(np.diag(h), device="cuda") for o in occ]
        self.D = (occ[0] * torch.tensor(U, device="cuda")) @ occ[1].T + one[0][:, None] + one[1][None, :]

    @staticmethod
    def hopping(h, b):
        row, col, val = [np.zeros(0, np.int64)], [np.zeros(0, np.int64)], [np.zeros(0)]
        for i, j in zip(*np.nonzero(h - np.diag(np.diag(h)))):
            r = np.nonzero(((b >> i) & 1) & ~(b >> j) & 1)[0]
            between = ((1 << max(i, j)) - 1) & ~((2 << min(i, j)) - 1)
            row.append(r)
            col.append(np.searchsorted(b, b[r] ^ (1 << int(i)) ^ (1 << int(j))))
            val.append(h[i, j] * (1.0 - 2.0 * (bits(b[r] & between) % 2)))
        at = torch.tensor(np.stack([np.concatenate(row), np.concatenate(col)]), device="cuda")
        return torch.sparse_coo_tensor(at, torch.tensor(np.concatenate(val), device="cuda"), (len(b), len(b))).to_sparse_csr()

    def __call__(self, x):
        y = self.D * x
        y += self.K[0] @ x
        y += (self.K[1] @ x.T.contiguous()).T
        return y


def lanczos(H, v, steps):
    """(V, alpha, beta, |v|) of the fully reorthogonalized recursion from v."""
    b0 = torch.linalg.vector_norm(v)
    V = torch.empty((steps, v.numel()), dtype=torch.float64, device="cuda")
    alpha, beta = torch.zeros(steps, dtype=torch.float64, device="cuda"), torch.zeros(steps, dtype=torch.float64, device="cuda")
    V[0] = v.reshape(-1) / b0
    m = steps
    for k in range(steps):
        w = H(V[k].reshape(v.shape)).reshape(-1)
        alpha[k] = torch.dot(V[k], w)
        for _ in range(2):
            w = w - V[:k + 1].T @ (V[:k + 1] @ w)
        beta[k] = torch.linalg.vector_norm(w)
        if k % 16 == 15 and float(beta[max(0, k - 15):k + 1].min()) < 1e-9:
            m = int((beta[:k + 1] < 1e-9).nonzero()[0]) + 1
            break
        if k + 1 < steps:
            V[k + 1] = w / beta[k]
    m = min(m, v.numel())
    return V[:m], alpha[:m].cpu().numpy(), beta[:m].cpu().numpy(), float(b0)


def tridiagonal(alpha, beta):
    return np.linalg.eigh(np.diag(alpha) + np.diag(beta[:-1], 1) + np.diag(beta[:-1], -1))


def ground(H, shape):
    v = torch.randn(shape, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    for _ in range(4):  # restarted until the residual is at rounding
        V, a, b, _ = lanczos(H, v, min(160, v.numel()))
        E, S = tridiagonal(a, b)
        v = (torch.tensor(S[:, 0], device="cuda") @ V).reshape(shape)
        v = v / torch.linalg.vector_norm(v)
        E0 = float(torch.sum(v * H(v)))
        if float(torch.linalg.vector_norm(H(v) - E0 * v)) < 1e-12 * max(1.0, abs(E0)):
            break
    return E0, v


def annihilated(c, psi, B, spin, create, i):
    """c+_i or c_i applied to psi for one spin; the basis of the other spin stays."""
    L = one_body(c).shape[0]
    n = (c["n_up"], c["n_dn"])[spin] + (1 if create else -1)
    T = spin_basis(L, n)
    ok = np.nonzero(((T >> i) & 1) == (1 if create else 0))[0]
    src = np.searchsorted(B[spin], T[ok] ^ (1 << i))
    sign = 1.0 - 2.0 * ((bits(T[ok] & ((1 << i) - 1)) + (c["n_up"] if spin else 0)) % 2)
    if spin == 1:
        psi = psi.T
    out = torch.zeros((len(T), psi.shape[1]), dtype=torch.float64, device="cuda")
    out[torch.tensor(ok, device="cuda")] = torch.tensor(sign, device="cuda")[:, None] * psi[torch.tensor(src, device="cuda")]
    return out.T.contiguous() if spin == 1 else out


def green(c, E0, psi, B, z, steps, spin=0):
    ns, L = c["t"].shape[0], one_body(c).shape[0]
    G = np.zeros((len(z), ns, ns), dtype=np.complex128)
    for create in (True, False):
        n = [c["n_up"], c["n_dn"]]
        n[spin] += 1 if create else -1
        if not 0 <= n[spin] <= L:
            continue
        H = Sector(c, *n)
        phi = [annihilated(c, psi, B, spin, create, i) for i in range(ns)]
        P = torch.stack([p.reshape(-1) for p in phi])
        if P.shape[1] <= 1300:
            eye = [torch.eye(len(b), dtype=torch.float64, device="cuda") for b in H.B]
            dense = torch.kron(H.K[0].to_dense(), eye[1]) + torch.kron(eye[0], H.K[1].to_dense()) + torch.diag(H.D.reshape(-1))
            E, S = np.linalg.eigh(dense.cpu().numpy())
            q = P.cpu().numpy() @ S
            w = 1.0 / (z[:, None] - (E - E0 if create else E0 - E)[None, :])
            G += np.einsum("zr,ir,jr->zij", w, q, q, optimize=True)
            continue
        for j in range(ns):
            if float(torch.linalg.vector_norm(phi[j])) < 1e-13:
                continue
            V, a, b, b0 = lanczos(H, phi[j], min(steps, phi[j].numel()))
            E, S = tridiagonal(a, b)
            q = (P @ V.T).cpu().numpy() @ S
            G[:, :, j] += (1.0 / (z[:, None] - (E - E0 if create else E0 - E)[None, :]) * (b0 * S[0])[None, :]) @ q.T
    return G


def exact(case, seed):
    kind = case["kind"]
    if kind == "hpsi":
        c = make_cluster(case["cluster"], case["size"], case["n_up"], case["n_dn"], seed)
        H = Sector(c, case["n_up"], case["n_dn"])
        du, dd = H.D.shape
        return H(hpsi_vector(case, seed, du, dd)[:, :dd].double().contiguous())
    if kind == "lattice":
        return exact_lattice(case, seed)
    if kind == "batch":
        E0, G = [], []
        for c in batch_clusters(case, seed):
            H = Sector(c, c["n_up"], c["n_dn"])
            e, psi = ground(H, H.D.shape)
            E0.append(e)
            if case["max_orb"] <= 7:  # sectors small enough for the dense form
                up = green(c, e, psi, H.B, complex_grid(case), 0)
                G.append(np.stack([up, up if c["n_up"] == c["n_dn"] else green(c, e, psi, H.B, complex_grid(case), 0, spin=1)]))
        return dict(E0=np.array(E0), G=by_sites(G) if G else None)
    if kind == "ground":
        c = make_cluster(case["cluster"], case["size"], case["n_up"], case["n_dn"], seed)
        if math.comb(orbitals(case["cluster"], case["size"]), case["n_up"]) > 1000:
            return None
        H = Sector(c, case["n_up"], case["n_dn"])
        return dict(E0=ground(H, H.D.shape)[0], vector=None)
    c = solve_cluster(case, seed) if kind == "solve" else sym_cluster(case, seed)[0]
    H = Sector(c, c["n_up"], c["n_dn"])
    if H.D.numel() > 1000000:
        return None
    E0, psi = ground(H, H.D.shape)
    z = complex_grid(case)
    return dict(E0=E0, G=green(c, E0, psi, H.B, z, 240 if case.get("matsubara", True) else 1200))


def complex_grid(case):
    return 1j * grid(case) if case.get("matsubara", True) else grid(case) + 1j * ETA


def exact_lattice(case, seed):
    s = lattice_inputs(case, seed)
    t = lambda a: torch.tensor(a, dtype=torch.complex128, device="cuda")  # noqa: E731
    L, lat = case["width"] * case["height"], s["lat"]
    E = np.asarray(lat["E"], dtype=np.float64)

    def V(kt):
        v = np.zeros((len(kt), L, L), dtype=np.complex128)
        for i, j, n, hop in lat["bonds"]:
            phase = np.exp(1j * kt @ (np.asarray(n, dtype=np.float64) @ E))
            v[:, i, j] += hop * phase
            v[:, j, i] += hop * phase.conj()
        return t(v)

    base = torch.linalg.inv(t(s["Gc"])) + t(s["Gamma"])
    phase = t(np.exp(-1j * s["k_cpt"] @ np.asarray(lat["pos"]).T))
    Gk = torch.empty((len(s["k_cpt"]), len(s["z"])), dtype=torch.complex128, device="cuda")
    for k, v in enumerate(V(s["k_cpt"])):
        Gk[k] = torch.einsum("i,zij,j->z", phase[k], torch.linalg.inv(base - v), phase[k].conj()) / L
    Gbar = sum(torch.linalg.inv(base - v) for v in V(s["k_cdmft"])) / len(s["k_cdmft"])
    A = base - torch.linalg.inv(Gbar)
    theta, eps, z, w = t(s["trial"][0]), t(s["trial"][1]), t(s["z"]), t(s["weights"])
    g = 1.0 / (z[None, :, None] - eps[:, None, :])
    R = A[None] - torch.einsum("cia,cza,cja->czij", theta, g, theta)
    d = torch.einsum("z,czij->c", w, R * R.conj()).real
    g_eps = -2.0 * torch.einsum("z,czij,cia,cja,cza->ca", w, R.conj(), theta, theta, g * g).real
    g_theta = -2.0 * torch.einsum("z,czij,cja,cza->cia", w, R.conj() + R.conj().transpose(2, 3), theta, g).real
    grad = torch.cat([g_eps, g_theta.reshape(len(d), -1)], dim=1)
    return dict(G=Gk.cpu().numpy(), A=A.cpu().numpy(), d=d.cpu().numpy(), grad=grad.cpu().numpy())
