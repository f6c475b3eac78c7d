"""The Schrodinger workspace that a mesh keeps between calls: several host threads, bounded memory.

Calls of several threads on one mesh give what they give one after the other (bit for bit: the
block operators sum in a fixed order).
"""
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
