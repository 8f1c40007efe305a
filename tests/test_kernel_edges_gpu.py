"""The CUDA kernels at the sizes where they change form (edges of tiles, smallest and largest of a
range), against the CPU oracle."""

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


# The tridiagonal eigensolver: one level (sectors of one state), levels that are no multiple of its
# chunks, energies far below and above 1 (the entries are scaled by a power of two).  E0 is the
# Rayleigh quotient of the reconstructed state, within 1e-10 of the largest energy scale.
@pytest.mark.parametrize("L,n_up,n_dn", [(1, 1, 1), (2, 0, 2), (2, 1, 1), (4, 1, 2), (6, 3, 3), (7, 3, 4)])
@pytest.mark.parametrize("scale", [1e-7, 1.0, 1e6])
def test_ground_energy_over_scales(L, n_up, n_dn, scale):
    rng = np.random.default_rng(100 * L + n_up)
    c = W.random_cluster(rng, L, 0, n_up, n_dn)
    c = dict(c, t=c["t"] * scale, U=c["U"] * scale, mu=c["mu"] * scale)
    H = O.jw_hamiltonian_dense(_model(c), n_up, n_dn)
    E = np.linalg.eigvalsh(H)
    tol = 1e-10 * max(abs(E[0]), abs(E[-1])) + 1e-13
    with ed.Cluster(c, seed=5) as cl:
        assert abs(cl.ground_state()[1] - E[0]) <= tol
    assert abs(ed.ed_batch_solve([c], seed=5)[0][0] - E[0]) <= tol


# Batched inversions in groups of 2, 4, 8, 16 and 32 lanes: every width at its ends, on matrices that
# need row swaps (a cyclic permutation plus noise; condition number below 10, so rounding stays
# below 1e-13 relative), with counts that do not fill the last warp.
@pytest.mark.parametrize("L", [1, 2, 3, 4, 5, 8, 9, 16, 17, 32])
def test_cpt_group_widths(L):
    rng = np.random.default_rng(L)
    nz, nk = 7, 5
    lat = W.square_superlattice(L, 1, -0.1)
    kt = rng.uniform(-3, 3, (nk, 1))
    Ginv = np.roll(np.eye(L), 1, axis=0) * (2.0 + 1.0j) + 0.02 * (rng.standard_normal((nz, L, L)) + 1j)
    Gc = np.linalg.inv(Ginv)
    V = np.zeros((nk, L, L), dtype=complex)
    for i, j, n, t in lat["bonds"]:
        ph = np.exp(1j * kt[:, 0] * n[0] * lat["E"][0, 0])
        V[:, i, j] += t * ph
        V[:, j, i] += t * ph.conj()
    ref = np.linalg.inv(Ginv[None] - V[:, None])
    G = ed.ed_cpt_green(lat, Gc, kt)
    assert np.abs(G - ref).max() <= 1e-12
    assert np.abs(ed.ed_cpt_green(lat, Gc, kt, ed.ED_CPT_AVERAGE) - ref.mean(axis=0)).max() <= 1e-12
    e = np.exp(-1j * kt * lat["pos"][:, 0][None])
    per = np.einsum("ki,kzij,kj->kz", e, ref, e.conj()) / L
    assert np.abs(ed.ed_cpt_green(lat, Gc, kt, ed.ED_CPT_PERIODIZED) - per).max() <= 1e-12


@pytest.mark.parametrize("bad", [0.0, np.nan])
def test_cpt_refuses_singular(bad):
    lat = W.square_superlattice(2, 1, -0.1)
    Gc = np.full((3, 2, 2), bad, dtype=complex)
    with pytest.raises(ed.EDError):
        ed.ed_cpt_green(lat, Gc, np.zeros((1, 1)))


# Distance and gradient: one frequency slice per thread up to 32, parameter tiles beyond 256.
@pytest.mark.parametrize("L,nb,nc", [(1, 1, 1), (2, 3, 65), (4, 8, 3), (6, 40, 2), (32, 32, 1)])
def test_distance_gradient_tiles(L, nb, nc):
    rng = np.random.default_rng(L * nb)
    nz = 37
    z = 1j * W.matsubara_grid(nz)
    theta, eps = rng.standard_normal((nc, L, nb)), rng.standard_normal((nc, nb))
    A = rng.standard_normal((nz, L, L)) + 1j * rng.standard_normal((nz, L, L))
    w = rng.uniform(0.0, 1.0, nz)
    d, grad = ed.ed_cdmft_distance(theta, eps, z, w, A, grad=True)
    g = 1.0 / (z[None, :, None] - eps[:, None, :])
    R = A[None] - np.einsum("cia,cza,cja->czij", theta, g, theta, optimize=True)
    d_ref = np.einsum("z,czij->c", w, np.abs(R) ** 2)
    ge = -2 * np.einsum("z,czij,cia,cja,cza->ca", w, R.conj(), theta, theta, g * g, optimize=True).real
    gt = -2 * np.einsum("z,czij,cja,cza->cia", w, R.conj() + R.conj().transpose(0, 1, 3, 2), theta, g, optimize=True).real
    ref = np.concatenate([ge, gt.reshape(nc, -1)], axis=1)
    assert np.abs(d - d_ref).max() <= 1e-12 * np.abs(d_ref).max()
    assert np.abs(grad - ref).max() <= 1e-11 * np.abs(ref).max()


# Continued fractions: thread blocks of 64 and 128 frequencies, levels staged 128 at a time (300-state
# sectors run past their dimension), checks on every second frequency from 2,048 on.
@pytest.mark.parametrize("nz", [1, 63, 65, 129, 2100])
def test_continued_fraction_grid_edges(nz):
    c = W.random_cluster(np.random.default_rng(3), 6, 0, 3, 3)
    om = np.linspace(-6.0, 6.0, nz)
    ref = O.green_exact(_model(c), 3, 3, om + 0.05j)[0]
    with ed.Cluster(c, seed=5) as cl:
        assert np.abs(cl.green(om, 0.05) - ref).max() <= 1e-8
    G = ed.ed_batch_solve([c], omega=om, eta=0.05, seed=5)[4][0]
    assert np.abs(G[0] - ref).max() <= 1e-8 and np.abs(G[1] - ref).max() <= 1e-8


# Frequencies far outside the spectrum, where eight levels of the recurrences leave the range of FP64: G is
# 1/z there up to (spectrum / |z|), so z G is the unit matrix to the rounding of the norms.
@pytest.mark.parametrize("z", [1e20, 1e40, -1e60, 1e140])
@pytest.mark.parametrize("axis", [ed.ED_AXIS_REAL, ed.ED_AXIS_MATSUBARA])
def test_continued_fraction_far_frequencies(z, axis):
    c = W.random_cluster(np.random.default_rng(3), 6, 0, 3, 3)
    zz = z + 0.05j if axis == ed.ED_AXIS_REAL else 1j * z
    om = np.array([0.5, z])
    with ed.Cluster(c, seed=5) as cl:
        G = cl.green(om, 0.05, axis)
    B = ed.ed_batch_solve([c], omega=om, eta=0.05, axis=axis, seed=5)[4][0]
    for g in (G[1], B[0][1], B[1][1]):
        assert np.abs(zz * g - np.eye(6)).max() <= 1e-10


# One-pass H.psi: flat index below 192 columns, tiles of 4, 2 and 1 rows with ragged last tiles and
# column chunks, rows too long for shared memory; padded rows keep their padding.  FP64 within 1e-12
# and FP32 within 2e-5 of max|y| (the bounds of the parity tests).
@pytest.mark.parametrize("L,n_up,n_dn", [(2, 1, 1), (20, 1, 2), (21, 1, 2), (10, 5, 5), (12, 1, 6), (12, 6, 5), (16, 3, 8),
                                         (18, 1, 8), (24, 1, 6)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("pad", [0, 3])
def test_one_pass_hpsi_forms(L, n_up, n_dn, dtype, pad):
    rng = np.random.default_rng(L + n_up)
    c = W.random_cluster(rng, L, 0, n_up, n_dn, U=4.0 if pad else None, dense_t=L <= 12)
    op = O.sector_hamiltonian(_model(c), n_up, n_dn)
    with ed.Cluster(c) as cl:
        du, dd = ed.ed_sector_dims(cl.h, n_up, n_dn)
        x = rng.standard_normal((du, dd))
        xd = torch.zeros((du, dd + pad), dtype=dtype, device="cuda")
        xd[:, :dd] = torch.tensor(x, device="cuda")
        y = torch.full((du, dd + pad), 7.0, dtype=dtype, device="cuda")
        ed.ed_hpsi(cl.h, n_up, n_dn, ed.ED_FP64 if dtype == torch.float64 else ed.ED_FP32, xd.data_ptr(), y.data_ptr(),
                   dd + pad, torch.cuda.current_stream().cuda_stream)
        got = y.cpu().double().numpy()
    ref = O.apply_h(op, xd[:, :dd].cpu().double().numpy()).reshape(du, dd)
    tol = 1e-12 if dtype == torch.float64 else 2e-5
    assert np.abs(got[:, :dd] - ref).max() <= tol * np.abs(ref).max()
    assert np.all(got[:, dd:] == 7.0)


# The fused step of the one-pass forms through whole solves (E0 within 1e-10 of the oracle).
@pytest.mark.parametrize("L,n_up,n_dn", [(6, 1, 3), (10, 5, 4), (12, 2, 6)])
@pytest.mark.parametrize("precision", [ed.ED_FP64, ed.ED_FP32])
def test_one_pass_lanczos_forms(L, n_up, n_dn, precision):
    c = W.random_cluster(np.random.default_rng(L), L, 0, n_up, n_dn)
    E = O.ground_state(O.sector_hamiltonian(_model(c), n_up, n_dn))[0]
    with ed.Cluster(c, seed=5, precision=precision) as cl:
        assert abs(cl.ground_state()[1] - np.min(E)) <= 1e-10 * abs(np.min(E))


# Levels of small sectors in clusters of 1 to 8 blocks: sectors of a few states (most blocks own
# nothing) up to 1,225, both precisions, both spins.  FP64 within 1e-8 of the exact Lehmann sum, FP32
# vectors within 2e-4 (the bounds of the parity tests on the real axis at eta = 0.05).
@pytest.mark.parametrize("L,n_up,n_dn", [(2, 1, 1), (3, 1, 2), (5, 2, 3), (7, 3, 4)])
@pytest.mark.parametrize("precision,tol", [(ed.ED_FP64, 1e-8), (ed.ED_FP32, 2e-4)])
def test_small_sector_levels(L, n_up, n_dn, precision, tol):
    c = W.random_cluster(np.random.default_rng(7 * L), L, 0, n_up, n_dn)
    om = np.linspace(-8.0, 8.0, 101)
    with ed.Cluster(c, seed=5, precision=precision) as cl:
        for spin in (0, 1):
            ref = O.green_exact(_model(c), n_up, n_dn, om + 0.05j, spin=spin)[0]
            assert np.abs(cl.green(om, 0.05, spin=spin) - ref).max() <= tol


# Band Lanczos at every group width of the block continued fraction (2, 4, 8, 16 lanes) and every split of
# the Gram's warps (1, 4, 9 and 16 pair tiles), against the exact Lehmann sum (FP64, 1e-8).
@pytest.mark.parametrize("ns,nb,n_up,n_dn", [(1, 5, 3, 3), (2, 4, 3, 2), (3, 3, 3, 3), (5, 1, 2, 3), (8, 0, 2, 1), (9, 0, 1, 1),
                                             (14, 0, 1, 1)])
def test_band_widths(ns, nb, n_up, n_dn):
    c = W.random_cluster(np.random.default_rng(ns), ns, nb, n_up, n_dn)
    om = W.matsubara_grid(33)
    ref = O.green_exact(_model(c), n_up, n_dn, 1j * om)[0]
    with ed.Cluster(c, seed=5, gf_method=ed.ED_GF_BAND) as cl:
        assert np.abs(cl.green(om, 0.0, axis=ed.ED_AXIS_MATSUBARA) - ref).max() <= 1e-8


# CUDA-core Gram with shared pair tiles: sums of n products of unit normal numbers, compensated FP32
# (1e-6 of sum |x y|, the bound of the other Gram checks).
@pytest.mark.parametrize("nx,ny", [(1, 1), (4, 4), (5, 8), (8, 8), (9, 12), (12, 12)])
@pytest.mark.parametrize("n", [128, 128 * 1023])
def test_gram_split_tiles(nx, ny, n):
    g = torch.Generator("cuda").manual_seed(nx * ny)
    x = torch.randn((nx, n), dtype=torch.float32, device="cuda", generator=g)
    y = torch.randn((ny, n), dtype=torch.float32, device="cuda", generator=g)
    xy = torch.cat([x, y])
    got = ed.ed_gram_f32(xy.data_ptr(), nx, xy[nx:].data_ptr(), ny, n, n, 0)
    ref = (x.double() @ y.double().T).cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-6 * float((x.abs().double() @ y.abs().double().T).max())


# FP64 products with integer hop sums (sectors of 2^19 states and more with few hop magnitudes): odd
# dimensions and leading dimensions, and lines that leave the fixed point for the FP64 sums: one huge
# element, zero and denormal rows, a row scaled to 1e-290.  Every row within 1e-12 of the largest |H| |x| that
# feeds it, so small rows are held to their own scale.
@pytest.mark.parametrize("W_,n_up,n_dn", [(7, 6, 7), (6, 6, 7), (7, 8, 5)])
@pytest.mark.parametrize("pad", [0, 1])
def test_integer_hop_sums(W_, n_up, n_dn, pad):
    rng = np.random.default_rng(W_ + n_up)
    L = 2 * W_ + (1 if W_ == 6 else 0)
    if W_ == 6:  # 13-site chain, one magnitude
        c = W.random_cluster(rng, L, 0, n_up, n_dn, U=4.0)
    else:
        c = W.served_request(rng, sizes=(L,))
        c = dict(c, n_up=n_up, n_dn=n_dn, U=c["U"] if pad else rng.uniform(1, 9, L))
    op = O.sector_hamiltonian(_model(c), n_up, n_dn)
    with ed.Cluster(c) as cl:
        du, dd = ed.ed_sector_dims(cl.h, n_up, n_dn)
        x = rng.standard_normal((du, dd))
        x[3, 5] = 1e9
        x[7] = 0.0
        x[8] = 5e-310
        x[9] *= 1e-290
        xd = torch.zeros((du, dd + pad), dtype=torch.float64, device="cuda")
        xd[:, :dd] = torch.tensor(x, device="cuda")
        y = torch.full((du, dd + pad), 7.0, dtype=torch.float64, device="cuda")
        args = (cl.h, n_up, n_dn, ed.ED_FP64, xd.data_ptr(), y.data_ptr(), dd + pad, torch.cuda.current_stream().cuda_stream)
        ed.ed_hpsi(*args)
        got = y.cpu().numpy()
        xd[11, 2] = float("nan")
        xd[13, 4] = float("inf")
        ed.ed_hpsi(*args)
        bad = ~np.isfinite(y[:, :dd].cpu().numpy())
    ref = O.apply_h(op, x).reshape(du, dd)
    fed = O.apply_h(op, (np.abs(x) > 1e5) * 1.0).reshape(du, dd) != 0.0  # rows and columns of the huge element
    assert np.abs(got[:, :dd] - ref)[~fed].max() <= 1e-12 * np.abs(ref[~fed]).max()
    assert np.abs(got[:, :dd] - ref)[fed].max() <= 1e-12 * np.abs(ref).max()
    assert np.all(got[:, dd:] == 7.0)
    z = np.zeros((du, dd))
    z[11, 2] = z[13, 4] = 1.0
    assert np.array_equal(bad, (O.apply_h(op, z).reshape(du, dd) != 0.0) | (z != 0.0))


# The two-pass kernels on tables ordered on the device (from 2,048 states per spin), with few and with
# many hop values (FP64: more than four magnitudes keep them off the integer sums).
@pytest.mark.parametrize("dtype,many", [(torch.float32, False), (torch.float32, True), (torch.float64, True)])
@pytest.mark.parametrize("n_up,n_dn", [(7, 7), (5, 8)])
def test_two_pass_ordered_tables(dtype, many, n_up, n_dn):
    rng = np.random.default_rng(n_up)
    c = W.served_request(rng, sizes=(14,))
    t = c["t"] * np.triu(rng.uniform(0.5, 1.5, c["t"].shape), 1) if many else np.triu(c["t"], 1)
    c = dict(c, t=t + t.T, n_up=n_up, n_dn=n_dn)
    op = O.sector_hamiltonian(_model(c), n_up, n_dn)
    with ed.Cluster(c) as cl:
        du, dd = ed.ed_sector_dims(cl.h, n_up, n_dn)
        ld = (dd + 127) // 128 * 128
        x = torch.zeros((du, ld), dtype=dtype, device="cuda")
        x[:, :dd] = torch.tensor(rng.standard_normal((du, dd)), device="cuda")
        y = torch.zeros_like(x)
        ed.ed_hpsi(cl.h, n_up, n_dn, ed.ED_FP64 if dtype == torch.float64 else ed.ED_FP32, x.data_ptr(), y.data_ptr(), ld,
                   torch.cuda.current_stream().cuda_stream)
        got = y.cpu().double().numpy()
    ref = O.apply_h(op, x[:, :dd].cpu().double().numpy()).reshape(du, dd)
    assert np.abs(got[:, :dd] - ref).max() <= (1e-12 if dtype == torch.float64 else 2e-5) * np.abs(ref).max()
    assert np.all(got[:, dd:] == 0.0)


# Lanczos vectors written straight into their store, in the forced two-pass form, both precisions.
@pytest.mark.parametrize("precision", [ed.ED_FP64, ed.ED_FP32])
def test_two_pass_ground_state_store(precision):
    c = W.random_cluster(np.random.default_rng(8), 10, 0, 5, 4)
    E = O.ground_state(O.sector_hamiltonian(_model(c), 5, 4))[0]
    with ed.Cluster(c, seed=5, precision=precision) as cl:
        ed.ed_set_option(cl.h, ed.ED_OPT_TWO_PASS_MIN_BYTES, 0.0)
        st, E0, res, _ = cl.ground_state()
        assert st == ed.ED_OK and res <= 1e-12 and abs(E0 - E) <= 1e-10 * abs(E)
