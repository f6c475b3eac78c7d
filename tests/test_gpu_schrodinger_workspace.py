"""The Schrodinger workspace that a mesh keeps between calls: several host threads, bounded memory; a
subdomain of as many planes as a mesh may have.

Calls of several threads on one mesh give what they give one after the other (bit for bit: the
block operators sum in a fixed order).
"""
import math
import threading

import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

M_EFF = (0.19, 0.19, 0.19)


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1403_7561_gb300 as qcad
    return qcad


def interior(dev):
    s = dev["subdomain"]
    return (s["i1"] - s["i0"] - 1) * (s["j1"] - s["j0"] - 1) * (s["k1"] - s["k0"] - 1)


def test_block_applies_of_several_threads(q):
    dev = W.five_gate_device(n=(64, 64, 48), T=4.0)
    n = interior(dev)
    m = q.qcad_mesh_create(dev)
    gen = torch.Generator(device="cuda").manual_seed(1)
    jobs = []
    for nvec in (1, 3, 8, 16):
        X = torch.randn(nvec, n, generator=gen, dtype=torch.float64, device="cuda")
        phi = torch.full((m.n_nodes,), -0.01 * nvec, dtype=torch.float64, device="cuda")
        jobs.append((phi, X, torch.empty_like(X), torch.empty_like(X)))
    torch.cuda.synchronize()
    for phi, X, HX, MX in jobs:
        q.qcad_schrodinger_apply(m, dev["bias"], phi, M_EFF, X, HX, MX)
    want = [(HX.clone(), MX.clone()) for _, _, HX, MX in jobs]
    torch.cuda.synchronize()
    fresh = q.qcad_mesh_create(dev)  # its workspace grows while the threads use it
    errors = []

    def work(k):
        phi, X, HX, MX = jobs[k]
        try:
            for _ in range(10):
                HX.fill_(float("nan"))
                MX.fill_(float("nan"))
                torch.cuda.synchronize()
                q.qcad_schrodinger_apply(fresh, dev["bias"], phi, M_EFF, X, HX, MX)
                if not (torch.equal(HX, want[k][0]) and torch.equal(MX, want[k][1])):
                    errors.append("thread %d: results differ" % k)
        except Exception as e:  # noqa: BLE001 - reported by the main thread
            errors.append("thread %d: %r" % (k, e))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def held(q, call):
    """Device bytes that a call leaves allocated (torch's own stay in its pool)."""
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    call()
    torch.cuda.synchronize()
    return before - torch.cuda.mem_get_info()[0]


def test_a_wide_block_apply_gives_its_memory_back(q):
    # 400 vectors on 65 x 65 x 33 nodes take 1.3 GB of block vectors; 1 GiB stays at most
    dev = W.five_gate_device(n=(128, 128, 96), T=4.0)
    m = q.qcad_mesh_create(dev)
    phi = torch.zeros(m.n_nodes, dtype=torch.float64, device="cuda")
    X = torch.ones(400, interior(dev), dtype=torch.float64, device="cuda")
    HX, M1 = torch.empty_like(X), torch.empty_like(X[:1])
    H1 = torch.empty_like(M1)
    q.qcad_schrodinger_apply(m, dev["bias"], phi, M_EFF, X[:1].contiguous(), H1, M1)
    assert held(q, lambda: q.qcad_schrodinger_apply(m, dev["bias"], phi, M_EFF, X, HX)) <= (1 << 30) + (4 << 20)
    assert torch.equal(HX[399], H1[0])
    q.qcad_schrodinger_apply(m, dev["bias"], phi, M_EFF, X[:1].contiguous(), H1, M1)  # after the release
    assert torch.equal(HX[0], H1[0])


def test_an_eigensolve_holds_what_its_rows_take(q):
    # per subdomain node: rows in FP32 and in double-float or FP64 (27 x 12 B), potential coefficients (64 B),
    # Jacobi scale and mask (9 B); the assembly's 64 MB; 2 MB pages of nine buffers
    dev = W.five_gate_device(n=(256, 256, 128), T=0.5)
    s = dev["subdomain"]
    nodes = (s["i1"] - s["i0"] + 1) * (s["j1"] - s["j0"] + 1) * (s["k1"] - s["k0"] + 1)
    small = W.five_gate_device(n=(64, 64, 48), T=0.5)  # loads the kernels
    ms = q.qcad_mesh_create(small)
    q.qcad_schrodinger_eigs(ms, small["bias"], torch.zeros(ms.n_nodes, dtype=torch.float64, device="cuda"), nev=2,
                            m_eff=M_EFF, tol=1e-6)
    m = q.qcad_mesh_create(dev)
    phi = torch.zeros(m.n_nodes, dtype=torch.float64, device="cuda")
    bytes_ = held(q, lambda: q.qcad_schrodinger_eigs(m, dev["bias"], phi, nev=2, m_eff=M_EFF, tol=1e-6))
    assert bytes_ <= 397 * nodes + (64 << 20) + 9 * (2 << 20)


def test_a_subdomain_of_65536_planes(q):
    # columns of one interior node by 63 and by 65534, layers of 1.5 nm: the lowest levels differ by the z
    # energy of 64 layers, kappa 6 (1 - cos t) / ((2 + cos t) h^2) with t = pi / 64 (the other one's is 2e-10 eV)
    E = {}
    for nz in (64, 65535):
        dev = dict(Lx=200.0, Ly=200.0, nx=2, ny=2, layers=[dict(material=0, thickness=1.5 * nz, n=nz)],
                   materials=[dict(W.SI)], gates=[], gate_work_function=None, bottom_ohmic=1, dots=[],
                   subdomain=dict(i0=0, i1=2, j0=0, j1=2, k0=0, k1=nz))
        m = q.qcad_mesh_create(dev)
        bias = dict(T=4.0, V_gate=[], V_sub=0.0, statistics=1, incomplete_ionization=1)
        phi = torch.zeros(m.n_nodes, dtype=torch.float64, device="cuda")
        E[nz] = q.qcad_schrodinger_eigs(m, bias, phi, nev=1, m_eff=M_EFF, tol=1e-8)[0][0]
    kappa, c = 0.0380998 / 0.19, math.cos(math.pi / 64)
    assert abs(E[64] - E[65535] - kappa * 6 * (1 - c) / ((2 + c) * 1.5 ** 2)) < 1e-7
