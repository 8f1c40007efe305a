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
