"""The cluster kernel at every kind of size it lays out: padded rows and
columns of open chains, rings whose rows and columns divide exactly, one to
many CTAs a cluster with idle warps in the last, every order up to the pairs
of middle stages, unaligned buffers, samples inside a launch; and the rings
that go to the tiles.  Compared with the per-term path (same FP32 Horner
stages, one launch each)."""
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


def _run(ctqw, w, flags=0, shift=0):
    h = ctqw.build_for_workload(w)
    n = h.total_amplitudes
    rng = np.random.default_rng(5)
    v = (rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64)
    v /= np.linalg.norm(v) / np.sqrt(w.R)
    psi = torch.zeros(n + shift, dtype=torch.complex64, device="cuda")[shift:]
    psi.copy_(torch.from_numpy(v))
    n_obs = h.n_obs(w.n_steps, w.obs_every)
    P, nr, en = ctqw._outputs(h, n_obs, True, True, True, "cuda")
    ws = torch.empty(3 * 8 * n + 8 * shift, dtype=torch.uint8, device="cuda")[8 * shift:]
    ctqw.ctqw_propagate_taylor(h, psi, w.dtype, w.dt, w.K, w.n_steps, w.obs_every, P, nr, en, flags=flags, workspace=ws)
    ctqw.ctqw_check_status(h)
    out = [psi.cpu().numpy()] + [t.cpu().numpy() for t in (P, nr, en) if t is not None]
    h.close()
    return out


def _check(ctqw, w, shift=0):
    a, b = _run(ctqw, w, shift=shift), _run(ctqw, w, flags=ctqw.FLAG_PLAIN, shift=shift)
    # amplitudes of norm-1 states; a step's increment (norm <= 0.3) carries a
    # few roundings of 2^-24 per stage: seven steps of up to 20 stages stay
    # below 7 * 0.3 * 20 * 2^-24 = 2.5e-6 in the norm of a state
    for r in range(w.R):
        n = len(a[0]) // w.R
        assert np.linalg.norm(a[0][r * n:(r + 1) * n] - b[0][r * n:(r + 1) * n]) <= 2.5e-6
    for x, y in zip(a[1:], b[1:]):   # P and norms to twice that, energies times ||H|| <= 12
        assert np.max(np.abs(x - y)) <= 12 * 5e-6


@pytest.mark.parametrize("N", [2, 3, 5, 31, 32, 33, 63, 65, 97, 100, 127, 129, 130, 191, 193, 250, 255])
@pytest.mark.parametrize("K", [1, 2, 3, 4, 16])
def test_open_chains(ctqw, N, K):
    w = cw.get("bosons_n256_u2").with_(N=N, R=3, K=K, n_steps=7, obs_every=2)
    _check(ctqw, w)


@pytest.mark.parametrize("N", [4, 12, 36, 64, 68, 100, 128, 132, 144, 192, 200, 248, 256, 6, 30, 98, 140, 99, 181])
def test_rings(ctqw, N):
    w = cw.get("bosons_n256_u2").with_(N=N, R=3, K=5, n_steps=7, obs_every=3, periodic=True, seed=4)
    _check(ctqw, w)


@pytest.mark.parametrize("N,R", [(20, 700), (100, 200), (196, 40), (256, 40)])
def test_more_realizations_than_clusters(ctqw, N, R):
    w = cw.get("bosons_n256_u2").with_(N=N, R=R, K=6, n_steps=3, obs_every=1)
    _check(ctqw, w)


@pytest.mark.parametrize("N", [48, 77, 100, 160, 256])
def test_unaligned_buffers(ctqw, N):
    w = cw.get("bosons_n256_u2").with_(N=N, R=3, K=7, n_steps=5, obs_every=2)
    _check(ctqw, w, shift=1)


def test_new_sizes_still_need_a_workspace(ctqw):
    w = cw.get("bosons_n256_u2").with_(N=100, R=2)
    h = ctqw.build_for_workload(w)
    psi = h.new_state(w.dtype)
    with pytest.raises(ctqw.CtqwError) as e:
        ctqw.ctqw_propagate_taylor(h, psi, w.dtype, w.dt, 8, 1)
    assert e.value.status == ctqw.CTQW_EINVAL
    h.close()


@pytest.mark.parametrize("N,R,periodic", [(30, 5, False), (64, 3, True), (100, 90, True), (130, 3, False), (256, 20, False)])
@pytest.mark.parametrize("every", [0, 1, 4])
def test_switching_in_the_kernel(ctqw, N, R, periodic, every):
    # the same law and draws as the per-term path, whose updates are launches of their own
    w = cw.get("bosons_n256_u2").with_(N=N, R=R, K=6, n_steps=9, periodic=periodic, sites=(N // 2 - 1, N // 2))
    got = {}
    for flags in (0, ctqw.FLAG_PLAIN):
        h = ctqw.build_for_workload(w)
        psi = h.new_state(w.dtype)
        ctqw.ctqw_init_state(h, psi, ctqw.initial_sites(w, h), w.dtype)
        P, nr, en = ctqw._outputs(h, h.n_obs(w.n_steps, every), True, True, True, "cuda")
        ctqw.ctqw_propagate_taylor_switching(h, psi, w.dtype, w.dt, w.K, w.n_steps, every, P, nr, en, 11, 0.2, flags)
        ctqw.ctqw_check_status(h)
        got[flags] = [psi.cpu().numpy()] + [t.cpu().numpy() for t in (P, nr, en) if t is not None] + list(h.params())
        h.close()
    a, b = got[0], got[ctqw.FLAG_PLAIN]
    assert np.array_equal(a[-1], b[-1]) and np.array_equal(a[-2], b[-2])   # parameters: the same bits
    for x, y in zip(a[:-2], b[:-2]):
        assert np.max(np.abs(x - y)) <= 12 * 5e-6
