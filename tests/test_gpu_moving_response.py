"""Calls on one mesh while the charge response moves between them.

The mesh keeps the activity map of the last linearization and the response states of its multigrid
elements; both follow the potential. Two biases in turn, whose carriers sit under different gates,
give on one mesh what they give on fresh meshes: J v bit for bit (no sum over the mesh enters it),
solutions within the solver's tolerance.
"""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

BIASES = ([0.7, 0.2, 0.7, 0.2, 0.2], [0.2, 0.2, 0.2, 0.2, 0.75], [0.1, 0.7, 0.1, 0.7, 0.1])


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1403_7561_gb300 as qcad
    return qcad


@pytest.mark.parametrize("n", [(64, 64, 48), (61, 45, 38)])
def test_two_biases_in_turn(q, n):
    dev = W.five_gate_device(n=n, T=4.0, with_subdomain=False)
    biases = [dict(dev["bias"], V_gate=V) for V in BIASES]
    new = lambda m: torch.zeros(m.n_nodes, dtype=torch.float64, device="cuda")  # noqa: E731

    def calls(m, bias, phi):
        out = []
        g = torch.Generator(device="cuda").manual_seed(2)
        v = torch.randn(m.n_nodes, generator=g, dtype=torch.float64, device="cuda")
        v[:(n[0] + 1) * (n[1] + 1)] = 0.0   # Dirichlet nodes: the contact below, the gates on top
        v[-(n[0] + 1) * (n[1] + 1):] = 0.0
        for precision in (0, 1):
            y = new(m)
            q.qcad_poisson_jv(m, bias, phi, v, y, precision)
            out.append(y)
        return out

    def solve(m, bias, precision):
        phi = new(m)
        q.qcad_poisson_solve(m, bias, q.make_opts(precision=precision, cheb_degree=-1), phi)
        return phi

    fresh_phi = [[solve(q.qcad_mesh_create(dev), b, p) for p in (0, 1)] for b in biases]
    fresh = [calls(q.qcad_mesh_create(dev), b, f[0]) for b, f in zip(biases, fresh_phi)]
    assert not torch.equal(fresh[0][0], fresh[1][0])
    m = q.qcad_mesh_create(dev)
    for k in (0, 1, 0, 2, 1):
        for p in (0, 1):
            assert torch.max(torch.abs(solve(m, biases[k], p) - fresh_phi[k][p])).item() <= 1e-9, (k, p)
        for got, want in zip(calls(m, biases[k], fresh_phi[k][0]), fresh[k]):
            assert torch.equal(got, want), k
