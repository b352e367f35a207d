"""Two-particle FP32 batches of more sizes than one launch of the register tiles
lists: sizes that share their tile counts, and more tile counts than that,
against the per-term path."""
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


def _run(ctqw, sizes, K, flags):
    R = len(sizes)
    rng = np.random.default_rng(3)
    n = int(np.sum(sizes))
    h = ctqw.Hamiltonian(2, 1, False, np.asarray(sizes, dtype=np.int32), 1.0, 1.0, 0.5, 0.25, rng.random(n),
                         rng.random(n))   # one bond draw a site, the wrap bond's unused
    g = torch.Generator("cuda").manual_seed(2)
    v = torch.view_as_complex(torch.randn(h.total_amplitudes, 2, generator=g, device="cuda"))
    for r in range(R):
        a, b = int(h.st_off[r]), int(h.st_off[r + 1])
        v[a:b] /= torch.linalg.vector_norm(v[a:b])
    P, nr, en = ctqw._outputs(h, h.n_obs(2, 1), True, True, True, "cuda")
    ctqw.ctqw_propagate_taylor(h, v, cw.C64, 0.02, K, 2, 1, P, nr, en, flags, h.workspace(cw.C64))
    ctqw.ctqw_check_status(h)
    out = [t.cpu().numpy() for t in (v, P, nr, en)]
    h.close()
    return out


@pytest.mark.parametrize("sizes,K", [(list(range(2, 90)), 8), ([700 - 7 * (i % 41) for i in range(60)], 5),
                                     (list(range(1960, 20, -44)), 7), (list(range(1700, 24, -36)), 4)])
def test_many_sizes(ctqw, sizes, K):
    a, b = _run(ctqw, sizes, K, 0), _run(ctqw, sizes, K, ctqw.FLAG_PLAIN)
    # norm-1 states, increments of norm <= 0.02 x 7 = 0.15 a step with a few
    # roundings of 2^-24 per stage: two steps below 2 x 0.15 x 16 x 2^-24 = 3e-7
    # a realization
    assert np.linalg.norm(a[0] - b[0]) <= 3e-7 * np.sqrt(len(sizes))
    for x, y in zip(a[1:], b[1:]):   # energies: times 2 ||H|| <= 14
        assert np.max(np.abs(x - y)) <= 14 * 3e-7
