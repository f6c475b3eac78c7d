"""The launch autotuner times the operator that the solves at the given bias run."""
import ctypes

import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1403_7561_gb300 as qcad
    return qcad


def test_time_follows_the_response(q):
    # at 300 K every silicon element responds to the potential, at 0.5 K those under the gates and at the
    # contact alone. An FP64 node plane with response takes five times the operations of one without
    ms = {}
    for T in (300.0, 0.5):
        dev = W.five_gate_device(n=(96, 96, 64), T=T, with_subdomain=False)
        m = q.qcad_mesh_create(dev)
        ms[T] = q.qcad_autotune(m, dev["bias"], 0)[3]
    assert ms[0.5] < 0.8 * ms[300.0], ms


@pytest.mark.parametrize("precision", [0, 1])
def test_solves_after_tuning(q, precision):
    # the same potential as with the default shapes, with and without a bias that can be solved
    dev = W.five_gate_device(n=(37, 33, 21), T=4.0, with_subdomain=False)
    opts = q.make_opts(precision=precision, cheb_degree=-1)
    phis = []
    for tune in (None, dev["bias"], dict(dev["bias"], V_gate=[0.0])):
        m = q.qcad_mesh_create(dev)
        if tune is not None:
            variant, rows, chunk, t = q.qcad_autotune(m, tune, precision)
            assert t > 0 and q.qcad_launch_info(m, 2 if precision else 1)[:3] == (variant, rows, chunk)
        phi = torch.zeros(m.n_nodes, dtype=torch.float64, device="cuda")
        q.qcad_poisson_solve(m, dev["bias"], opts, phi)
        phis.append(phi)
    for phi in phis[1:]:
        assert torch.max(torch.abs(phi - phis[0])).item() <= 1e-9


def test_a_bias_that_cannot_be_solved_tunes_as_none(q):
    # no voltages, no temperature, no bias at all: the shapes are timed with response everywhere
    dev = W.five_gate_device(n=(37, 33, 21), T=4.0, with_subdomain=False)
    m = q.qcad_mesh_create(dev)
    no_voltages, no_temperature = q.make_bias(dev["bias"]), q.make_bias(dict(dev["bias"], T=0.0))
    no_voltages.V_gate = ctypes.POINTER(ctypes.c_double)()
    t = ctypes.c_float()
    for b in (ctypes.byref(no_voltages), ctypes.byref(no_temperature), None):
        assert q._lib.qcad_autotune(m.handle, b, 1, None, None, None, ctypes.byref(t)) == 0
        assert t.value > 0
