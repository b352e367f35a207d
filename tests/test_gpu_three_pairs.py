"""Three particles, two Horner stages per launch: rings and open chains from
lattices smaller than a block's rows to the largest side, odd and even orders,
samples, ragged batches and switching noise, against the per-term path."""
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


def _run(ctqw, w, flags, switch):
    h = ctqw.build_for_workload(w)
    g = torch.Generator("cuda").manual_seed(2)
    v = torch.view_as_complex(torch.randn(h.total_amplitudes, 2, generator=g, device="cuda"))
    for r in range(w.R):
        a, b = int(h.st_off[r]), int(h.st_off[r + 1])
        v[a:b] /= torch.linalg.vector_norm(v[a:b])
    P, nr, en = ctqw._outputs(h, h.n_obs(w.n_steps, w.obs_every), True, True, True, "cuda")
    if switch:
        ctqw.ctqw_propagate_taylor_switching(h, v, w.dtype, w.dt, w.K, w.n_steps, w.obs_every, P, nr, en, 5, 0.3, flags)
    else:
        ctqw.ctqw_propagate_taylor(h, v, w.dtype, w.dt, w.K, w.n_steps, w.obs_every, P, nr, en, flags, h.workspace(w.dtype))
    ctqw.ctqw_check_status(h)
    out = [t.cpu().numpy() for t in (v, P, nr, en)]
    h.close()
    return out


def _check(ctqw, w, switch=False):
    a, b = _run(ctqw, w, 0, switch), _run(ctqw, w, ctqw.FLAG_PLAIN, switch)
    # norm-1 states, increments of norm <= 0.2 a step with a few roundings of
    # 2^-24 per stage: five steps below 5 * 0.2 * 16 * 2^-24 = 1e-6 a realization
    assert np.linalg.norm(a[0] - b[0]) <= 1e-6 * np.sqrt(w.R)
    for x, y in zip(a[1:], b[1:]):   # energies: times 2 ||H|| <= 24
        assert np.max(np.abs(x - y)) <= 24e-6


@pytest.mark.parametrize("N", [2, 3, 5, 12, 16, 31, 47, 64, 97, 160, 213])
@pytest.mark.parametrize("K,periodic", [(1, True), (2, False), (5, True), (8, False)])
def test_uniform(ctqw, N, K, periodic):
    w = cw.get("ring3_n160").with_(N=N, R=2, K=K, n_steps=5, obs_every=2, periodic=periodic, J_halfwidth=0.25,
                                   sites=(0, 0, 1))
    _check(ctqw, w)


@pytest.mark.parametrize("switch", [False, True])
def test_ragged(ctqw, switch):
    w = cw.get("ring3_n160").with_(N=40, R=7, K=6, n_steps=5, obs_every=1, ragged_sizes=(9, 24, 33, 40), J_halfwidth=0.25,
                                   sites=(0, 0, 1))
    _check(ctqw, w, switch)
