"""Rings of a few sites, which only the tiles take among the two-particle FP32
paths: RK4 on few and on many realizations (tiles and stages), and two sites,
whose tiles copy one amplitude at a time."""
import numpy as np
import pytest

import ctqw_workloads as cw
from gpu_helpers import U_FP32, h_bound, oracle_params

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


def _h(eps, J, U):
    N = len(eps)
    H1 = np.diag(eps)
    for i in range(N):   # at N = 2 both bonds join the same sites
        H1[i, (i + 1) % N] -= J[i]
        H1[(i + 1) % N, i] -= J[i]
    H = np.kron(H1, np.eye(N)) + np.kron(np.eye(N), H1)
    return H + U * np.diag(np.eye(N).reshape(-1))


@pytest.mark.parametrize("N", [2, 3, 6, 14, 22])
@pytest.mark.parametrize("R", [5, 460, 1300])
@pytest.mark.parametrize("K", [4, 7])   # 4: RK4
def test_against_sums(ctqw, N, R, K):
    w = cw.get("bosons_n256_u2").with_(N=N, R=R, K=K, periodic=True, sites=(0, 1), n_steps=3)
    h = ctqw.build_for_workload(w)
    rng = np.random.default_rng(N * R)
    v = rng.standard_normal((R, N * N)) + 1j * rng.standard_normal((R, N * N))
    v = (v / np.linalg.norm(v, axis=1, keepdims=True)).astype(np.complex64)
    psi = torch.from_numpy(v.reshape(-1)).cuda()
    nr = torch.empty((2, R), dtype=torch.float64, device="cuda")
    if K == 4:
        ctqw.ctqw_propagate_rk4(h, psi, cw.C64, w.dt, 3, 2, None, nr, None, 0, h.workspace(cw.C64, ctqw.RK4))
    else:
        ctqw.ctqw_propagate_taylor(h, psi, cw.C64, w.dt, K, 3, 2, None, nr, None, 0, h.workspace(cw.C64))
    ctqw.ctqw_check_status(h)
    got = psi.cpu().numpy().reshape(R, -1)
    h.close()
    # a step rounds its stages relative to dt ||H|| and the state by an ulp or
    # two (the stages' update is not compensated)
    hd = w.dt * h_bound(w)
    tol = 3 * (16 * hd * np.exp(hd) + 4) * U_FP32
    some = [0, R // 2, R - 1]
    for r, (eps, J) in zip(some, oracle_params(w, some)):
        A = -1j * w.dt * _h(eps, J, w.U)
        ref = v[r].astype(np.complex128)
        for _ in range(3):
            t = ref
            for j in range(1, K + 1):
                t = A @ t / j
                ref = ref + t
        assert np.linalg.norm(got[r] - ref) <= tol
