"""Switching noise on the cluster kernel with few stages a launch: orders 1, 2
and 6 with a sample, and so a launch, after every step.  A cluster's first CTA
stores the redrawn parameters where the other CTAs of the cluster have read the
old ones; with few stages nothing but the barrier after the reads keeps the two
apart.  States that are spread over the whole lattice, so that every CTA's
coefficients count, against the oracle's steps in FP64."""
import numpy as np
import pytest

import ctqw_workloads as cw
import oracle
from gpu_helpers import U_FP32, h_bound

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SEED, P_SWITCH = 0xC0FFEE, 1.0


@pytest.fixture(scope="module")
def ctqw():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1612_00746_gb300 import build, ctqw as c

    build.build()
    c.load()
    return c


def _oracle(w, r, psi):
    N = w.N
    ue, uj = cw.uniform_draws(w.seed, [r], [N])
    eps, J = oracle.workload_parameters(w, ue[0], uj[0], N)
    for n in range(w.n_steps):
        H = oracle.many_particle_hamiltonian(oracle.single_particle_hamiltonian(eps, J, w.periodic), w.m, w.U)
        psi = oracle.taylor_step(H, psi, w.dt, w.K)
        eps, J = oracle.switch_parameters(eps, J, r, n, SEED, P_SWITCH, N, w.periodic, 0.0, w.eps_halfwidth, w.J0,
                                          w.J_halfwidth)
    return psi, eps, J


# (orders of 12 and more a launch run on the clusters at these sizes, the
# lower ones on the tiles)
@pytest.mark.parametrize("K", [1, 2, 6, 12, 14])
@pytest.mark.parametrize("N,R,steps", [(256, 1, 6), (256, 4, 4), (256, 20, 2), (128, 3, 4), (200, 2, 4)])
def test_a_launch_after_every_step(ctqw, N, R, steps, K):
    w = cw.get("bosons_n256_u2").with_(N=N, R=R, K=K, n_steps=steps, obs_every=1, sites=(N // 2 - 1, N // 2))
    rng = np.random.default_rng(N + R)
    v = rng.standard_normal((R, N * N)) + 1j * rng.standard_normal((R, N * N))
    v = (v / np.linalg.norm(v, axis=1, keepdims=True)).astype(np.complex64)
    h = ctqw.build_for_workload(w)
    psi = torch.from_numpy(v.reshape(-1)).cuda()
    P, nr, en = ctqw._outputs(h, h.n_obs(steps, 1), True, True, True, "cuda")
    ctqw.ctqw_propagate_taylor_switching(h, psi, cw.C64, w.dt, K, steps, 1, P, nr, en, SEED, P_SWITCH)
    ctqw.ctqw_check_status(h)
    got, (eps, J) = psi.cpu().numpy().reshape(R, N * N), h.params()
    h.close()
    # a stage rounds each of its six products, sums and coefficients a few
    # times, all of them relative to dt ||H||: 16 U dt ||H|| e^(dt ||H||) a step,
    # and half an ulp a step for the state itself
    hd = w.dt * h_bound(w)
    tol = steps * (16 * hd * np.exp(hd) + 1) * U_FP32
    for r in range(R):
        ref, e_ref, J_ref = _oracle(w, r, v[r].astype(np.complex128))
        assert np.linalg.norm(got[r] - ref) <= tol
        assert np.array_equal(eps[r * N:(r + 1) * N], e_ref)
        assert np.array_equal(J[r * N:r * N + N - 1], np.asarray(J_ref)[:N - 1])
