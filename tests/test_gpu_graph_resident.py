"""Two particles on small graphs in FP32: the on-chip path over node counts and
degrees at the edges of its blocks (one and two columns a thread, one CTA and
clusters, rows of another CTA, padded rows, repeated links, no links at all),
few and many realizations, chunks, orders and samples, against the FP64 path of
the same handle."""
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


def _links(kind, n):
    i = np.arange(n)
    if kind == "none":
        return i[:0], i[:0]
    if kind == "chain":
        return i[:-1], i[1:]
    if kind == "torus":      # n = a b
        a = next(d for d in range(int(n ** 0.5), 0, -1) if n % d == 0)
        x = i.reshape(a, n // a)
        return np.concatenate([i, i]), np.concatenate([np.roll(x, -1, 0).ravel(), np.roll(x, -1, 1).ravel()])
    if kind == "double":     # every link of a ring twice
        return np.concatenate([i, i]), np.concatenate([(i + 1) % n, (i + 1) % n])
    if kind == "star":       # one node of many links, above 8 from n = 10
        return np.zeros(n - 1, dtype=int), i[1:]
    deg = int(kind[1:])      # ring with chords, degree as given
    steps = [1 + (n // 3 * k) % (n // 2 - 1) for k in range(deg // 2)]
    return np.concatenate([i] * len(steps)), np.concatenate([(i + s) % n for s in steps])


CASES = [("chain", 2, 1, 0, 1), ("none", 5, 3, 0, 3), ("torus", 9, 1500, 0, 7), ("chain", 31, 5, 0, 2), ("chain", 32, 6, 4, 9),
         ("double", 33, 130, 0, 6), ("d6", 40, 7, 0, 8), ("torus", 64, 700, 0, 12), ("d8", 65, 37, 8, 5), ("torus", 96, 2, 0, 16),
         ("star", 20, 9, 0, 6), ("torus", 119, 33, 0, 4), ("torus", 120, 160, 0, 8), ("d4", 166, 21, 12, 11), ("torus", 225, 1, 0, 16),
         ("torus", 225, 150, 0, 3), ("d6", 225, 5, 0, 10), ("torus", 256, 40, 0, 9), ("torus", 323, 12, 0, 6), ("torus", 400, 9, 0, 8),
         ("chain", 460, 3, 0, 5), ("torus", 480, 2, 0, 5)]


@pytest.mark.parametrize("kind,n,R,chunk,K", CASES)
def test_graph_on_chip(ctqw, kind, n, R, chunk, K):
    u, v = _links(kind, n)
    rng = np.random.default_rng(n)
    g = ctqw.Graph(2, 1, n, u, v, R, 1.0, 1.5, 0.5, 0.25, rng.random((R, n)), rng.random((R, len(u))))
    if chunk:
        ctqw.ctqw_graph_set_chunk(g, chunk)
    steps, every, dt = 6, 4, 0.02 if K > 2 else 0.002
    gen = torch.Generator("cuda").manual_seed(1)
    x = torch.view_as_complex(torch.randn(g.D, g.Rp, 2, generator=gen, device="cuda", dtype=torch.float64))
    x /= torch.linalg.vector_norm(x, dim=0)
    x[:, R:] = 0
    out = []
    for dtype in (cw.C64, cw.C128):
        psi = g.new_state(dtype, torch.device("cuda", 0))
        psi.copy_(x.reshape(psi.shape).to(torch.complex64))   # the same start for both
        n_obs = g.n_obs(steps, every)
        P = torch.empty((n_obs, n), dtype=torch.float64, device="cuda")
        nr = torch.empty((n_obs, R), dtype=torch.float64, device="cuda")
        en = torch.empty((n_obs, R), dtype=torch.float64, device="cuda")
        ctqw.ctqw_graph_propagate_taylor(g, psi, dtype, dt, K, steps, every, P, nr, en)
        out.append([t.cpu().numpy() for t in (torch.view_as_real(psi).double(), P, nr, en)])
    g.close()
    # Per step the increment dt |H| <= 0.02 (8 x 1.25 x 2 + 2.5) = 0.45 is formed
    # with 2 x 8 + 6 roundings of 2^-24 a stage, the stages' own errors shrinking
    # as dt |H| / j: 6 steps x 0.45 x 22 x 2^-24 x e^0.45 < 6e-6 of the norm, 1,
    # and the star's |H| (sqrt 19 x 1.25 x 2 + 2.5 = 14) is smaller; the final
    # rounding of psi is 2^-24.
    a, b = out
    assert np.max(np.abs(a[0] - b[0])) <= 6e-6
    # sums of squares of amplitudes with that error (2 |psi| |dpsi|), the norm 1;
    # energies of magnitude |H| <= 22.5
    assert np.max(np.abs(a[1] - b[1])) <= 1.2e-5
    assert np.max(np.abs(a[2] - b[2])) <= 1.2e-5
    assert np.max(np.abs(a[3] - b[3])) <= 22.5 * 1.2e-5 + 22.5 * 2 ** -22
    assert a[0].reshape(g.D, g.Rp, 2)[:, R:].any() == np.False_   # padding realizations stay zero
