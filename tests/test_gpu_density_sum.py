"""The sum of the tensor-core density's partial results keeps what an FP64 sum
keeps: contributions whose exact sum has 53 significant bits, one a split."""
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


@pytest.mark.parametrize("N", [64, 128, 256])
@pytest.mark.parametrize("order", [(0, 4, 8), (8, 4, 0), (4, 0, 8), (1, 2, 3), (0, 21, 63)])
def test_sum_of_the_splits(ctqw, N, order):
    R = 64   # 1 / (R m) is a power of two: the scale rounds nothing
    w = cw.get("bosons_n256_u2").with_(N=N, R=R, sites=(N // 2 - 1, N // 2))
    h = ctqw.build_for_workload(w)
    psi = np.zeros((R, N, N), dtype=np.complex64)
    x, y = N - 3, 5
    # |psi|^2 = 1, 2^-26, 2^-52 of both particles on x: products and single
    # contributions are exact, their sum has 53 bits, and so every FP64 sum of
    # them is exact in any order
    for r, e in zip(order, (0, -13, -26)):
        psi[r, x, x] = 2.0 ** e
    # Im: the same numbers off the diagonal, psi(x, k) conj(psi(y, k)) = i |.|^2 for k = 1
    for r, e in zip(order, (0, -13, -26)):
        psi[r, x, 1] = 1j * 2.0 ** e
        psi[r, y, 1] = 2.0 ** e
    rho = ctqw.ctqw_one_body_density(h, torch.from_numpy(psi.reshape(-1)).cuda(), cw.C64)[0].cpu().numpy()
    ctqw.ctqw_check_status(h)
    h.close()
    s = (1.0 + 2.0 ** -26) + 2.0 ** -52
    assert s - 1.0 - 2.0 ** -26 == 2.0 ** -52
    assert rho[x, y] == 1j * s / (2 * R) and rho[y, x] == -1j * s / (2 * R)
    # x holds the pair (both particles) and the single one at (x, 1): 2 s + s,
    # 54 bits, so half an ulp of the sum
    assert abs(rho[x, x].real - 3.0 * s / (2 * R)) <= 2.0 ** -53 * 4 / (2 * R) and rho[x, x].imag == 0.0
