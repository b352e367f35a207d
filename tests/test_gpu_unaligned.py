"""FP32 states that start off a 16-byte boundary, as a view into a larger buffer
may: the density matrix takes the kernel that reads one amplitude at a time, and
the kernels that read pairs and have no such form refuse the call."""
import numpy as np
import pytest

import ctqw_workloads as cw

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctqw():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1612_00746_gb300 import build, ctqw as c

    build.build()
    c.load()
    return c


def _state(total, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    v = torch.randn(2 * (total + 1), device="cuda", generator=gen).view(torch.complex64)
    return (v / v.abs().pow(2).sum().sqrt())[1:]


@pytest.mark.parametrize("N,R", [(16, 5), (64, 3), (256, 2)])
def test_density(ctqw, N, R):
    w = cw.get("bosons_n256_u2").with_(N=N, R=R, sites=(N // 2 - 1, N // 2))
    h = ctqw.build_for_workload(w)
    psi = _state(h.total_amplitudes, N)
    assert psi.data_ptr() % 16 == 8
    rho = ctqw.ctqw_one_body_density(h, psi, cw.C64)[0].cpu().numpy()
    ctqw.ctqw_check_status(h)
    p = psi.cpu().numpy().astype(np.complex128).reshape(R, N, N)
    ref = sum(a @ a.conj().T + a.T @ a.conj() for a in p) / (2 * R)
    # FP32 products summed over 32 k, then FP64: the CUDA-core kernel's bound
    assert np.max(np.abs(rho - ref)) <= 2e-6 * np.max(np.abs(ref))
    h.close()


def _refused(ctqw, call):
    with pytest.raises(ctqw.CtqwError) as e:
        call()
    assert e.value.status == ctqw.CTQW_EINVAL and "16-byte" in str(e.value)


@pytest.mark.parametrize("shape", [4, 8])
def test_pair_layouts_refuse(ctqw, shape):
    w = cw.get("bosons_n256_u2").with_(N=64, R=2, K=8, sites=(31, 32))
    h = ctqw.build_for_workload(w)
    ws = torch.empty(3 * 8 * h.total_amplitudes, dtype=torch.uint8, device="cuda")
    _refused(ctqw, lambda: ctqw.ctqw_propagate_taylor(h, _state(h.total_amplitudes, 1), cw.C64, w.dt, 8, 1, 0, None,
                                                      None, None, ctqw.FUSED_SHAPE(shape), ws))
    h.close()


def test_graphs_refuse(ctqw):
    w = cw.get_graph("lattice2d_15x15_m2").with_(R=5)
    g = ctqw.Graph.from_workload(w)
    psi = _state(g.total_amplitudes, 2)
    ws = g.workspace(cw.C64)
    nr = torch.empty((2, g.R), dtype=torch.float64, device="cuda")
    _refused(ctqw, lambda: ctqw.ctqw_graph_observables(g, psi, cw.C64, None, nr[0], None))
    _refused(ctqw, lambda: ctqw.ctqw_graph_propagate_taylor(g, psi, cw.C64, w.dt, 4, 1, 1, None, nr, None, ws))
    _refused(ctqw, lambda: ctqw.ctqw_graph_propagate_rk4(g, psi, cw.C64, w.dt, 1, 0, None, None, None, ws))
    g.close()
