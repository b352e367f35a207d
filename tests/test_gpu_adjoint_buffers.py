"""The adjoint chains' 16-byte and 8-byte copies: the gradient from buffers on
and off a 16-byte boundary, even and odd lattice sides and depths, with and
without interaction."""
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


@pytest.mark.parametrize("N,periodic", [(33, False), (48, True), (64, True), (97, False), (130, True)])
@pytest.mark.parametrize("K,U", [(4, 1.0), (5, 0.0), (7, 2.0), (14, 0.0), (16, 1.0)])
def test_unaligned_buffers_give_the_same_bits(ctqw, N, periodic, K, U):
    # the same arithmetic on the same values, summed in a fixed order: equal to
    # the last bit
    w = cw.get("bosons_n256_u2").with_(N=N, R=3, periodic=periodic, K=K, U=U, J_halfwidth=0.2, sites=(N // 2 - 1, N // 2))
    out = []
    for shift in (0, 1):
        h = ctqw.build_for_workload(w)
        psi = torch.zeros(h.total_amplitudes + shift, dtype=torch.complex64, device="cuda")[shift:]
        ctqw.ctqw_init_state(h, psi, ctqw.initial_sites(w, h), cw.C64)
        size = ctqw.adjoint_workspace(h, cw.C64, K, 5, 2).numel()
        ws = torch.empty(size + 8 * shift, dtype=torch.uint8, device="cuda")[8 * shift:]
        target = torch.full((h.p_width,), 1.0 / N, dtype=torch.float64)
        got = ctqw.ctqw_adjoint_grad(h, psi, cw.C64, 0.02, K, 5, 2, target, workspace=ws)
        # the gradients; the loss and the final occupation are sums of FP64
        # atomics, in no fixed order
        out.append([got[k].cpu().numpy() for k in (1, 2, 4, 5)])
        h.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
