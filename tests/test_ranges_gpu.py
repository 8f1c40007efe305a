"""The kernels at the ends of what their entry points take, and in the forms that options select."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle as O
from paper_2305_18643_gb300 import build, ed
from paper_2305_18643_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def libed():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    return ed.lib()


def _model(c):
    return O.Model(c["t"], c["U"], c["mu"], c["eps"], c["theta"])


def _product(cl, n_up, n_dn, x, ld):
    """ed_hpsi on an FP64 vector with leading dimension ld."""
    du, dd = x.shape
    xd = torch.zeros((du, ld), dtype=torch.float64, device="cuda")
    xd[:, :dd] = torch.tensor(x, device="cuda")
    y = torch.zeros_like(xd)
    ed.ed_hpsi(cl.h, n_up, n_dn, ed.ED_FP64, xd.data_ptr(), y.data_ptr(), ld, torch.cuda.current_stream().cuda_stream)
    return y[:, :dd].cpu().numpy()


# FP64 products are accurate element by element: every y[u, d] is a sum of at most 64 products in FP64, so it is
# within 64 2^-53 of (|H| |x|)[u, d] (times two for the reference's own rounding), however small it is
# beside the rest of its row and column.  Vectors: columns at 1e-10 of the others (a column and all that it hops
# to, so that sums of small operands alone occur), elements over 30 decades, and everything near 1e-290.
@pytest.mark.parametrize("kind", ["small columns", "thirty decades", "tiny"])
@pytest.mark.parametrize("n_up,n_dn,padded", [(6, 7, True), (6, 7, False), (5, 8, True), (4, 5, False)])
def test_fp64_products_element_by_element(kind, n_up, n_dn, padded):
    rng = np.random.default_rng(n_up)
    c = dict(W.served_request(rng, sizes=(14,)), n_up=n_up, n_dn=n_dn)
    op = O.sector_hamiltonian(_model(c), n_up, n_dn)
    du, dd = op.shape2
    x = rng.standard_normal((du, dd))
    if kind == "small columns":
        for d0 in (0, dd // 2):
            x[:, np.append(op.K_dn[d0].indices, d0)] *= 1e-10
    elif kind == "thirty decades":
        x *= 10.0 ** rng.uniform(-30.0, 0.0, (du, dd))
    else:
        x *= 1e-290
    with ed.Cluster(c) as cl:
        got = _product(cl, n_up, n_dn, x, (dd + 127) // 128 * 128 if padded else dd)
    bound = abs(op.K_up) @ abs(x) + (abs(op.K_dn) @ abs(x).T).T + abs(op.V) * abs(x)
    assert np.all(np.abs(got - O.apply_h(op, x)) <= 2 * 64 * 2.0 ** -53 * bound)


def _launches(fn):
    n = ed.ed_launch_count()
    fn()
    return ed.ed_launch_count() - n


# ED_OPT_TWO_PASS_MIN_BYTES selects the form of every product: two launches with 0, one beyond every size.
@pytest.mark.parametrize("dtype", [ed.ED_FP64, ed.ED_FP32])
@pytest.mark.parametrize("L,n_up,n_dn", [(8, 4, 4), (13, 6, 7)])
def test_two_pass_option_selects_the_product(L, n_up, n_dn, dtype):
    c = dict(W.served_request(np.random.default_rng(1), sizes=(8,)) if L == 8 else
             W.random_cluster(np.random.default_rng(1), L, 0, n_up, n_dn, U=4.0), n_up=n_up, n_dn=n_dn)
    with ed.Cluster(c) as cl:
        du, dd = ed.ed_sector_dims(cl.h, n_up, n_dn)
        ld = (dd + 127) // 128 * 128
        x = torch.zeros((du, ld), dtype=torch.float64 if dtype == ed.ED_FP64 else torch.float32, device="cuda")
        y = torch.zeros_like(x)
        for value, launches in ((0.0, 2), (9.1e18, 1)):
            ed.ed_set_option(cl.h, ed.ED_OPT_TWO_PASS_MIN_BYTES, value)
            assert _launches(lambda: ed.ed_hpsi(cl.h, n_up, n_dn, dtype, x.data_ptr(), y.data_ptr(), ld,
                                                torch.cuda.current_stream().cuda_stream)) == launches


# A forced two-pass form holds for continued fractions too (row pass, column pass and normalization per
# level), and gives the G of the form that small sectors take by themselves, at sectors from a few states
# up to and past the largest of the cluster kernel (1e-8, 2e-4 with FP32 vectors: the bounds of the parity tests).
@pytest.mark.parametrize("L,n_up,n_dn", [(2, 1, 1), (8, 4, 4), (9, 4, 4), (12, 3, 2), (9, 4, 5), (17, 2, 2)])
@pytest.mark.parametrize("precision,tol", [(ed.ED_FP64, 1e-8), (ed.ED_FP32, 2e-4)])
def test_two_pass_option_selects_the_fractions(L, n_up, n_dn, precision, tol):
    c = W.random_cluster(np.random.default_rng(L), L, 0, n_up, n_dn)
    om = W.matsubara_grid(65)
    G = []
    for force in (False, True):
        with ed.Cluster(c, seed=5, precision=precision) as cl:
            if force:
                ed.ed_set_option(cl.h, ed.ED_OPT_TWO_PASS_MIN_BYTES, 0)
            cl.ground_state()
            n = _launches(lambda: G.append(cl.green(om, 0.0, axis=ed.ED_AXIS_MATSUBARA)))
            longest = ed.ed_green_stats(cl.h)[1]
    assert n >= 3 * longest
    assert np.abs(G[0] - G[1]).max() <= tol


# Continued fractions of clusters whose energies are far beyond the frequencies: eight levels of the recurrences leave
# the range of FP64 by the coefficients alone.  Within 1e-8 of the largest |G| of the exact Lehmann sum.
@pytest.mark.parametrize("scale", [2.0 ** 40, 2.0 ** 130, 2.0 ** 200])
def test_continued_fraction_huge_energies(scale):
    c = W.random_cluster(np.random.default_rng(3), 6, 0, 3, 3)
    om = np.array([0.0, 0.5, -2.0])
    ref = O.green_exact(_model(c), 3, 3, (om + 0.05j) / scale)[0] / scale
    c = dict(c, t=c["t"] * scale, U=c["U"] * scale, mu=c["mu"] * scale)
    with ed.Cluster(c, seed=5) as cl:
        G = cl.green(om, 0.05)
    B = ed.ed_batch_solve([c], omega=om, eta=0.05, seed=5)[4][0]
    for g in (G, B[0], B[1]):
        assert np.abs(g - ref).max() <= 1e-8 * np.abs(ref).max()


# Band Lanczos of the same clusters: the Gram matrices hold the squares of the energies, beyond the range of FP32.
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 70, 2.0 ** 200])
@pytest.mark.parametrize("ns", [3, 8])
def test_band_huge_energies(scale, ns):
    c = W.random_cluster(np.random.default_rng(ns), ns, 0, 2, 1)
    om = W.matsubara_grid(17) * scale
    ref = O.green_exact(_model(c), 2, 1, 1j * om / scale)[0] / scale
    c = dict(c, t=c["t"] * scale, U=c["U"] * scale, mu=c["mu"] * scale)
    with ed.Cluster(c, seed=5, gf_method=ed.ED_GF_BAND) as cl:
        ed.ed_set_option(cl.h, ed.ED_OPT_GF_TOL, 1e-10 / scale)  # an absolute change of G
        G = cl.green(om, 0.0, axis=ed.ED_AXIS_MATSUBARA)
    assert np.abs(G - ref).max() <= 1e-8 * np.abs(ref).max()


# Matrices whose pivots' squares underflow are refused, not answered with infinities.
@pytest.mark.parametrize("L", [1, 2, 5, 17])
def test_cpt_refuses_underflowing_pivots(L):
    lat = W.square_superlattice(L, 1, -0.1)
    Gc = np.tile((np.eye(L) + 0.1j) * 1e-170, (3, 1, 1))
    with pytest.raises(ed.EDError):
        ed.ed_cpt_green(lat, Gc, np.zeros((1, 1)))


# The periodized G depends on differences of site positions alone: an origin at 2^33 lattice constants (where the
# positions are still exact) changes nothing.
def test_periodized_cpt_far_origin():
    rng = np.random.default_rng(2)
    lat = W.square_superlattice(2, 2, -1.0, 0.3)
    kt = rng.uniform(-3, 3, (9, 2))
    Gc = np.linalg.inv((2.0 + 1.0j) * np.eye(4) + 0.1 * rng.standard_normal((5, 4, 4)))
    G = ed.ed_cpt_green(lat, Gc, kt, ed.ED_CPT_PERIODIZED)
    far = ed.ed_cpt_green(dict(lat, pos=lat["pos"] + 2.0 ** 33), Gc, kt, ed.ED_CPT_PERIODIZED)
    assert np.abs(far - G).max() <= 1e-13 * np.abs(G).max()


@pytest.fixture(scope="module")
def tridiag(tmp_path_factory):
    here = os.path.dirname(os.path.abspath(__file__))
    so = str(tmp_path_factory.mktemp("tridiag") / "tridiag_reference.so")
    subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-shared", "-o", so, os.path.join(here, "tridiag_reference.cu")],
                   check=True)
    return ctypes.CDLL(so)


# Both eigenvalues, the eigenvector and the Ritz estimate bit for bit those of the plain form: random Lanczos
# coefficients, a chain broken into equal halves (a double lowest eigenvalue), a diagonal matrix, and Wilkinson's
# matrix (pairs of eigenvalues close together).
@pytest.mark.parametrize("kind", ["random", "halves", "diagonal", "wilkinson"])
@pytest.mark.parametrize("n", [1, 2, 3, 33, 600])
@pytest.mark.parametrize("threads", [64, 256])
def test_tridiagonal_bit_for_bit(tridiag, kind, n, threads):
    rng = np.random.default_rng(n)
    a, b = rng.standard_normal(n) - 3.0, rng.uniform(0.1, 3.0, n + 1)
    if kind == "halves":
        a[n // 2:n // 2 * 2], b[n // 2 + 1:n // 2 * 2] = a[:n // 2], b[1:n // 2]
        b[n // 2] = 0.0
    elif kind == "diagonal":
        b[:] = 0.0
    elif kind == "wilkinson":
        a, b = np.abs(np.arange(n) - (n - 1) / 2.0), np.ones(n + 1)
    for scale in (1e-7, 1.0, 1e6):
        ab = [torch.tensor(v * scale, device="cuda") for v in (a, b)]
        out = [torch.zeros(m, dtype=torch.float64, device="cuda") for m in (4, 2 * n, 4, 2 * n)]
        assert tridiag.tridiag_both(*[ctypes.c_void_p(t.data_ptr()) for t in ab], n, threads,
                                    *[ctypes.c_void_p(t.data_ptr()) for t in out]) == 0
        fast, vec, plain, ref = [t.cpu().numpy() for t in out]
        assert np.array_equal(fast[:3], plain[:3])
        assert np.array_equal(vec[:n], ref[:n])


# Solves keep their buffers in a pool while a cluster lives; the last one to go gives the memory back but for 512
# MiB.  A larger solve's own kernels take less than 16 MiB; the vectors of this one are 6.8 MB each.
@pytest.mark.parametrize("method", [ed.ED_GF_CF, ed.ED_GF_BAND])
def test_last_cluster_returns_its_memory(method):
    def solve(c):
        with ed.Cluster(W.hubbard_dimer(), seed=5) as other:
            with ed.Cluster(c, gf_method=method, seed=5) as cl:
                ed.ed_set_option(cl.h, ed.ED_OPT_GF_TOL, 1e-3)
                cl.green(W.matsubara_grid(8), 0.0, axis=ed.ED_AXIS_MATSUBARA)
            other.ground_state()
        return torch.cuda.mem_get_info()[0]

    free = solve(W.plain_2x4())
    assert solve(W.cdmft_2x2_bath()) >= free - (528 << 20)


# Rows too long for shared memory, dealt to the blocks in chunks of columns, in the fused step of a whole solve.
def test_long_rows_lanczos():
    c = W.random_cluster(np.random.default_rng(18), 18, 0, 1, 8)
    E = O.ground_state(O.sector_hamiltonian(_model(c), 1, 8))[0]
    with ed.Cluster(c, seed=5) as cl:
        assert abs(cl.ground_state()[1] - np.min(E)) <= 1e-10 * abs(np.min(E))


# The launches of a symmetrized Green function are counted and timed: beside every product of its runs there is
# a vector update, and every run is evaluated.
def test_symmetrized_fractions_are_counted():
    c, mirrors = W.open_3x4_c2v()
    kernels = {ed.ed_profile_kernel_name(k): k for k in range(11)}
    with ed.Cluster(dict(c, n_up=2, n_dn=1), seed=5) as cl:
        sym = ed.ed_sym_create(cl.h, mirrors, [1, 1])
        try:
            ed.ed_sym_ground_state(sym)
            ed.ed_profile_enable(True)
            ed.ed_sym_green(sym, W.matsubara_grid(16), 12, axis=ed.ED_AXIS_MATSUBARA)
            n = {k: ed.ed_profile_read(kernels[k])[0] for k in ("hpsi", "vector", "gf_eval")}
        finally:
            ed.ed_profile_enable(False)
            ed.ed_sym_destroy(sym)
    assert n["vector"] >= n["hpsi"] > 0 and n["gf_eval"] > 0


# Single FP32 rows that would fill an SM's shared memory take the same form (rows of 43,758).
def test_long_fp32_rows_lanczos():
    c = W.random_cluster(np.random.default_rng(18), 18, 0, 1, 8)
    with ed.Cluster(c, seed=5) as cl, ed.Cluster(c, seed=5, precision=ed.ED_FP32) as cl32:
        E = cl.ground_state()[1]
        assert abs(cl32.ground_state()[1] - E) <= 1e-10 * abs(E)
