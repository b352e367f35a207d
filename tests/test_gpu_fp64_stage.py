"""The FP64 Horner stage (rows walked in registers) at its edges: row blocks
of every length, columns around the 32- and 256-wide blocks, rings and open
chains, one-stage steps (the state updated from a copy), three particles, and
RK4 as the order-4 polynomial, against numpy in FP64."""
import numpy as np
import pytest

import ctqw_workloads as cw
from gpu_helpers import oracle_params

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
    m = psi.ndim
    y = np.zeros_like(psi)
    for a in range(m):
        sh = [1] * m
        sh[a] = -1
        y += eps.reshape(sh) * psi
        y -= J.reshape(sh) * np.roll(psi, -1, a) + np.roll(J, 1).reshape(sh) * np.roll(psi, 1, a)
    x = np.indices(psi.shape)
    for a in range(m):
        for b in range(a + 1, m):
            y += U * (x[a] == x[b]) * psi
    return y


def _compare(ctqw, w, method):
    rng = np.random.default_rng(1)
    h = ctqw.build_for_workload(w)
    psi0 = []
    for n in h.sizes:
        v = rng.standard_normal((int(n),) * w.m) + 1j * rng.standard_normal((int(n),) * w.m)
        psi0.append(v / np.linalg.norm(v))
    psi = torch.from_numpy(np.concatenate([v.reshape(-1) for v in psi0])).cuda()
    ws = h.workspace(w.dtype, method)
    if method == ctqw.TAYLOR:
        ctqw.ctqw_propagate_taylor(h, psi, w.dtype, w.dt, w.K, w.n_steps, workspace=ws)
    else:
        ctqw.ctqw_propagate_rk4(h, psi, w.dtype, w.dt, w.n_steps, workspace=ws)
    ctqw.ctqw_check_status(h)
    got = psi.cpu().numpy()
    K = w.K if method == ctqw.TAYLOR else 4
    for r, (eps, J) in enumerate(oracle_params(w)):
        ref = psi0[r]
        for _ in range(w.n_steps):
            phi, acc = ref, ref
            for j in range(1, K + 1):
                phi = -1j * w.dt / j * _apply(phi, eps, J, w.U)
                acc = acc + phi
            ref = acc
        # 3 steps of up to 20 terms, a few roundings of 2^-53 each on
        # amplitudes below 1: well inside 1e-14
        assert np.max(np.abs(got[h.st_off[r]:h.st_off[r + 1]] - ref.reshape(-1))) <= 1e-14
    h.close()


@pytest.mark.parametrize("N,R,periodic", [(2, 3, True), (3, 2, False), (31, 5, True), (33, 300, False), (64, 8, False),
                                          (100, 40, True), (255, 2, True), (257, 3, False), (300, 25, True)])
@pytest.mark.parametrize("K", [1, 2, 12])
def test_two_particles(ctqw, N, R, periodic, K):
    w = cw.get("bosons_n256_u2").with_(N=N, R=R, periodic=periodic, K=K, n_steps=3, dtype=cw.C128)
    _compare(ctqw, w, ctqw.TAYLOR)


@pytest.mark.parametrize("N,periodic", [(5, True), (13, False)])
def test_three_particles(ctqw, N, periodic):
    w = cw.get("ring3_n160").with_(N=N, R=3, periodic=periodic, K=7, n_steps=3, dtype=cw.C128, J_halfwidth=0.25)
    _compare(ctqw, w, ctqw.TAYLOR)


@pytest.mark.parametrize("N,R", [(9, 4), (70, 6)])
def test_ragged_and_rk4(ctqw, N, R):
    w = cw.get("ragged_n128_1024").with_(R=R, ragged_sizes=(N, N + 7, 2 * N), n_steps=3, dtype=cw.C128, sites=(-1, 0))
    _compare(ctqw, w, ctqw.TAYLOR)
    _compare(ctqw, w, ctqw.RK4)


@pytest.mark.parametrize("N,R", [(2, 1), (3, 2), (7, 5), (16, 1), (17, 3), (31, 4), (32, 70), (48, 9), (64, 8), (65, 2), (100, 1),
                                 (128, 1)])
@pytest.mark.parametrize("K,periodic", [(1, True), (5, False), (12, True)])
def test_resident_states(ctqw, N, R, K, periodic):
    # the sizes that stay on chip: slabs of one row, uneven last slabs, one
    # to eight amplitudes a thread; with samples (a launch per interval)
    w = cw.get("bosons_n256_u2").with_(N=N, R=R, periodic=periodic, K=K, n_steps=3, dtype=cw.C128)
    _compare(ctqw, w, ctqw.TAYLOR)
    h = ctqw.build_for_workload(w)
    out = []
    for flags in (0, ctqw.FLAG_PLAIN):
        psi = torch.randn(2 * h.total_amplitudes, dtype=torch.float64, device="cuda",
                          generator=torch.Generator("cuda").manual_seed(1)).view(torch.complex128) / N
        P, nr, en = ctqw._outputs(h, h.n_obs(5, 2), True, True, True, "cuda")
        ctqw.ctqw_propagate_taylor(h, psi, w.dtype, w.dt, K, 5, 2, P, nr, en, flags, h.workspace(w.dtype))
        out.append([t.cpu().numpy() for t in (psi, P, nr, en)])
    h.close()
    for a, b in zip(*out):   # sums of up to N^2 products of order 1 / N^2
        assert np.max(np.abs(a - b)) <= 1e-12
