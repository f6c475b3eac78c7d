"""Residual and Jacobian-vector product on grids where the default launch shapes are fitted.

Small grids take smaller tiles and z chunks than large ones (kernels_lin.cu fit_lin,
kernels_poisson.cu fit_march64); the sizes sit at the edges of tiles (30 columns, 2, 6 and 14 rows)
and of chunks. Against the oracle, with the tolerances of test_gpu_poisson.py: 1e-12 of the largest
entry in FP64, 2e-6 for the FP32 apply.
"""
import numpy as np
import pytest
import torch

import workloads as W
from oracle.poisson import PoissonProblem

pytestmark = pytest.mark.gpu

SIZES = [(16, 16, 32), (29, 13, 5), (30, 14, 33), (91, 3, 9), (7, 62, 4), (2, 2, 130)]


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1403_7561_gb300 as qcad
    return qcad


@pytest.mark.parametrize("T", [4.0, 300.0])
@pytest.mark.parametrize("n", SIZES)
def test_residual_and_jv_with_default_shapes(q, n, T):
    dev = W.five_gate_device(n=n, T=T, with_subdomain=False)
    P = PoissonProblem(dev)
    rng = np.random.default_rng(1)
    phi = P.initial_guess()
    phi[P.free] += 0.01 * rng.standard_normal(P.free.sum())
    v = rng.standard_normal(P.mesh.n_nodes)
    v[P.dir] = 0.0
    J = P.jacobian(phi)
    y0 = J @ v
    y0[P.dir] = 0.0
    R0 = P.residual(phi)
    d0 = np.where(P.dir, 1.0, J.diagonal())
    m = q.qcad_mesh_create(dev)
    t = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")  # noqa: E731
    R, D, y = (torch.full((m.n_nodes,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(3))
    q.qcad_poisson_residual(m, dev["bias"], t(phi), R, D)
    assert np.max(np.abs(R.cpu().numpy() - R0)) <= 1e-12 * np.max(np.abs(R0))
    assert np.max(np.abs(D.cpu().numpy() - d0)) <= 1e-12 * np.max(np.abs(d0))
    for precision, tol in ((0, 1e-12), (1, 2e-6)):
        q.qcad_poisson_jv(m, dev["bias"], t(phi), t(v), y, precision)
        assert np.max(np.abs(y.cpu().numpy() - y0)) <= tol * np.max(np.abs(y0)), precision


def test_residual_of_an_overflowing_density_is_infinite(q):
    # phi = 1e80 V: eta^4 exceeds the FP64 range and the Fermi-Dirac density with it. A constant phi has
    # K phi = 0, so every silicon node above the Ohmic contact holds the infinite charge alone
    dev = W.five_gate_device(n=(16, 16, 16), T=300.0, with_subdomain=False)
    m = q.qcad_mesh_create(dev)
    phi = torch.full((m.n_nodes,), 1e80, dtype=torch.float64, device="cuda")
    R = torch.zeros_like(phi)
    rmax, r2 = q.qcad_poisson_residual(m, dev["bias"], phi, R)
    n_si = dev["layers"][0]["n"]
    planes = R.cpu().numpy().reshape(-1, 17 * 17)
    assert np.all(planes[1:n_si + 1] == np.inf) and np.all(planes[0] == 0.0)
    assert rmax == np.inf and r2 == np.inf
