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
