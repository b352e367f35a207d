"""FP64 states on chip with six and eight amplitudes a thread, which many
realizations or large lattices take: odd sizes, uneven last slabs, several
CTAs an SM; and the four RK4 stages (which a call without the per-term flag no
longer runs) against the oracle's."""
import numpy as np
import pytest

import ctqw_workloads as cw
import oracle
from gpu_helpers import TOL_FP32, TOL_FP64, oracle_params

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


def _apply(psi, eps, J, U):
    y = (eps[:, None] + eps[None, :]) * psi + U * np.diag(np.diag(psi))
    left = np.roll(J, 1)
    for a in range(2):
        sh = (-1, 1) if a == 0 else (1, -1)
        y -= J.reshape(sh) * np.roll(psi, -1, a) + left.reshape(sh) * np.roll(psi, 1, a)
    return y


@pytest.mark.parametrize("N,R", [(65, 29), (100, 150), (149, 100), (81, 29), (170, 200), (176, 7)])
@pytest.mark.parametrize("K,periodic", [(1, True), (6, False), (7, True)])
def test_wide_threads(ctqw, N, R, K, periodic):
    w = cw.get("bosons_n256_u2").with_(N=N, R=R, periodic=periodic, K=K, n_steps=3, dtype=cw.C128,
                                       sites=(N // 2 - 1, N // 2))
    h = ctqw.build_for_workload(w)
    gen = torch.Generator("cuda").manual_seed(N)
    psi = torch.randn(2 * h.total_amplitudes, dtype=torch.float64, device="cuda", generator=gen).view(torch.complex128)
    psi = psi / N   # norms about sqrt(2)
    some = [0, R // 2, R - 1]
    start = {r: psi[r * N * N:(r + 1) * N * N].cpu().numpy().reshape(N, N) for r in some}
    ctqw.ctqw_propagate_taylor(h, psi, w.dtype, w.dt, K, 3, 0, None, None, None, 0, h.workspace(w.dtype))
    ctqw.ctqw_check_status(h)
    for r, (eps, J) in zip(some, oracle_params(w, some)):
        ref = start[r]
        for _ in range(3):
            phi = acc = ref
            for j in range(1, K + 1):
                phi = -1j * w.dt / j * _apply(phi, eps, J, w.U)
                acc = acc + phi
            ref = acc
        # 3 steps of up to 7 terms, a few roundings of 2^-53 each on
        # amplitudes below 1: well inside 1e-14
        assert np.max(np.abs(psi[r * N * N:(r + 1) * N * N].cpu().numpy().reshape(N, N) - ref)) <= 1e-14
    h.close()


@pytest.mark.parametrize("dtype,tol", [(cw.C128, TOL_FP64), (cw.C64, 50 * TOL_FP32)])
@pytest.mark.parametrize("name", ["bosons_small", "ring3_small"])
def test_the_four_stages(ctqw, name, dtype, tol):
    # in FP32 the plain RK4 update is not compensated: up to half an ulp of the
    # state a step beside the roundings that TOL_FP32 covers for one
    w = cw.get(name).with_(R=2, n_steps=50, obs_every=25, dtype=dtype)
    got = ctqw.run_workload(w, method=ctqw.RK4, flags=ctqw.FLAG_PLAIN)
    ref = oracle.ensemble_run(w, method="rk4")
    assert np.max(np.abs(got["P_mean"] - ref["P_mean"])) <= tol
    # and the default call, which runs the order-4 polynomial
    poly = ctqw.run_workload(w, method=ctqw.RK4)
    assert np.max(np.abs(poly["P_mean"] - got["P_mean"])) <= 2 * tol
