"""Block operators and block sizes of the eigensolver at the edges of their kernels.

H and M of 1 to 13 vectors (groups of 2 and 4 per thread, remainders) on subdomains that fit no
thread block, against the oracle's assembled operators (1e-12 of the largest entry in FP64, 2e-6 in
FP32, as in test_gpu_schrodinger_adjoint.py); eigenpairs for block sizes 3 to 20 (every width of the
update and Gram kernels) against the oracle's eigenvalues (1e-9 relative).
"""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import schrodinger as OS
from oracle.poisson import PoissonProblem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1403_7561_gb300 as qcad
    return qcad


def dt(a):
    return torch.tensor(np.asarray(a, dtype=np.float64), device="cuda")


@pytest.mark.parametrize("n", [(16, 18, 14), (37, 33, 21)])
@pytest.mark.parametrize("nvec", [1, 2, 4, 5, 13])
def test_hm_apply_block_sizes(q, n, nvec):
    dev = W.five_gate_device(n=n, T=4.0)
    P = PoissonProblem(dev)
    phi = P.initial_guess()
    me = (0.19, 0.21, 0.9)
    sel = P.mesh.subdomain_elements()
    H, M, idx = OS.operators(P.mesh, sel, P.mesh.subdomain_interior_nodes(), me, OS.device_potential(P, phi, sel))
    m = q.qcad_mesh_create(dev)
    X = np.random.default_rng(3).standard_normal((nvec, len(idx)))
    for precision, tol in ((0, 1e-12), (1, 2e-6)):
        HX = torch.full((nvec, len(idx)), float("nan"), dtype=torch.float64, device="cuda")
        MX = torch.full_like(HX, float("nan"))
        q.qcad_schrodinger_apply(m, dev["bias"], dt(phi), me, dt(X), HX, MX, precision)
        for j in range(nvec):
            ho, mo = H @ X[j], M @ X[j]
            assert np.max(np.abs(HX[j].cpu().numpy() - ho)) <= tol * np.max(np.abs(ho)), (precision, j)
            assert np.max(np.abs(MX[j].cpu().numpy() - mo)) <= tol * np.max(np.abs(mo)), (precision, j)


@pytest.mark.parametrize("nev", [1, 4, 7, 11, 16])
def test_eigenvalues_every_block_width(q, nev):
    dev = W.five_gate_device(n=(32, 32, 24), T=4.0)
    P = PoissonProblem(dev)
    phi = P.initial_guess()
    phi *= 0.3  # levels a few hundred meV above the Fermi level
    Eo = OS.solve_device(P, phi, nev=nev)[0]
    m = q.qcad_mesh_create(dev)
    E, rep = q.qcad_schrodinger_eigs(m, dev["bias"], dt(phi), nev=nev, tol=1e-8)
    assert rep["status"] == "OK", rep
    assert np.max(np.abs(np.array(E) - Eo) / np.abs(Eo)) < 1e-9
