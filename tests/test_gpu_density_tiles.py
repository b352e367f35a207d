"""The tensor-core density matrix over its ways of sharing the work: a diagonal
tile alone, off-diagonal tiles beside it, few and many realizations, two and
three particles, against the FP64 path on the same states."""
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


@pytest.mark.parametrize("m,N,R", [(2, 16, 1), (2, 16, 90), (2, 112, 3), (2, 128, 200), (2, 144, 1), (2, 256, 77), (2, 272, 5),
                                   (2, 400, 3), (2, 640, 2), (3, 16, 7), (3, 48, 3)])
def test_density_tiles(ctqw, m, N, R):
    w = cw.get("bosons_n256_u2" if m == 2 else "ring3_n160").with_(N=N, R=R, sites=(0,) * m)
    h = ctqw.build_for_workload(w)
    g = torch.Generator("cuda").manual_seed(N + R)
    x = torch.randn(h.total_amplitudes, 2, generator=g, device="cuda") / N ** (m / 2)
    psi = torch.view_as_complex(x)
    ctqw.ctqw_set_density_method(h, 0)
    a = ctqw.ctqw_one_body_density(h, psi, cw.C64)[0].cpu().numpy()
    ctqw.ctqw_check_status(h)
    b = ctqw.ctqw_one_body_density(h, psi.to(torch.complex128), cw.C128)[0].cpu().numpy()
    h.close()
    # FP32 sums over 256 k that may round toward zero: 256 x 2^-23 of the largest
    # element; the split operands and their dropped product 2^-21 of it
    assert np.max(np.abs(a - b)) <= (256 * 2.0 ** -23 + 2.0 ** -21) * np.max(np.abs(b))
    # Im of both triangles is one difference (Re of a diagonal tile adds hi lo
    # and lo hi in one order for both, so it is symmetric to rounding only)
    assert np.array_equal(a.imag, -a.imag.T)


@pytest.mark.parametrize("m,N,R", [(2, 5, 3), (2, 31, 9), (2, 33, 8), (2, 63, 2), (2, 65, 17), (2, 97, 1), (2, 130, 4), (3, 7, 5),
                                   (3, 19, 9), (3, 35, 2)])
def test_density_cuda_cores(ctqw, m, N, R):
    w = cw.get("bosons_n256_u2" if m == 2 else "ring3_n160").with_(N=N, R=R, sites=(0,) * m)
    h = ctqw.build_for_workload(w)
    g = torch.Generator("cuda").manual_seed(N + R)
    x = torch.randn(h.total_amplitudes, 2, generator=g, device="cuda") / N ** (m / 2)
    psi = torch.view_as_complex(x)
    v = psi.to(torch.complex128).reshape((R,) + (N,) * m)
    ref = 0
    for j in range(m):
        u = v.movedim(1 + j, 1).reshape(R, N, -1)
        ref = ref + torch.einsum("rxk,ryk->xy", u, u.conj())
    ref = (ref / (R * m)).cpu().numpy()
    ctqw.ctqw_set_density_method(h, 1)
    for dtype, state, tol in ((cw.C64, psi, 32 * 2.0 ** -24), (cw.C128, psi.to(torch.complex128), 1e-13)):
        a = ctqw.ctqw_one_body_density(h, state, dtype)[0].cpu().numpy()
        # FP32 sums of 32 products, each rounding 2^-24 of a sum of |terms| that
        # the largest element bounds; everything else in FP64
        assert np.max(np.abs(a - ref)) <= tol * np.max(np.abs(ref))
    h.close()
