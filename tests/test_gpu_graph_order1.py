"""Graphs at order 1 in FP32, where the only stage of a step reads the
neighbours of the state that it replaces: the stage path (graphs whose iterate
stays off chip: three particles, many links), whole and in chunks, and the path
on chip, against sums in FP64."""
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


def _graph(kind):
    rng = np.random.default_rng(3)
    if kind == "dense":      # up to 30 links a node
        return 2, 60, [(int(i), int(j)) for i in range(60) for j in rng.choice(60, 10, replace=False) if i != j]
    if kind == "three":
        return 3, 12, [(i, (i + 1) % 12) for i in range(12)]
    if kind == "large":      # two iterates of a realization do not fit on chip
        return 2, 700, [(i, (i + 1) % 700) for i in range(700)]
    return 2, 40, [(i, (i + 1) % 40) for i in range(40)]


def _apply(psi, H1, U, m):
    y = sum(np.moveaxis(np.tensordot(H1, psi, (1, a)), 0, a) for a in range(m))
    x = np.indices(psi.shape)
    for a in range(m):
        for b in range(a + 1, m):
            y = y + U * (x[a] == x[b]) * psi
    return y


@pytest.mark.parametrize("kind", ["dense", "three", "large", "ring"])
@pytest.mark.parametrize("every,chunk", [(0, 0), (1, 0), (1, 3)])
def test_order_one(ctqw, kind, every, chunk):
    m, N, edges = _graph(kind)
    R, steps, dt, U = 5, 4, 0.01, 2.0
    rng = np.random.default_rng(7)
    g = ctqw.Graph(m, 0, N, [e[0] for e in edges], [e[1] for e in edges], R, 1.0, U, 1.0, 0.25, rng.random((R, N)),
                   rng.random((R, len(edges))))
    if chunk:
        ctqw.ctqw_graph_set_chunk(g, chunk)
    eps, J = g.params()
    v = rng.standard_normal((R, N ** m)) + 1j * rng.standard_normal((R, N ** m))
    v = (v / np.linalg.norm(v, axis=1, keepdims=True)).astype(np.complex64)
    x = np.zeros((N ** m, g.Rp), dtype=np.complex64)
    x[:, :R] = v.T
    psi = torch.from_numpy(x.reshape(-1)).cuda()
    nr = torch.empty((steps + 1, R), dtype=torch.float64, device="cuda") if every else None
    ctqw.ctqw_graph_propagate_taylor(g, psi, cw.C64, dt, 1, steps, every, None, nr, None, g.workspace(cw.C64))
    torch.cuda.synchronize()
    got = psi.cpu().numpy().reshape(N ** m, g.Rp)[:, :R]
    g.close()
    links = np.bincount(np.array(edges).reshape(-1), minlength=N).max()
    # a step adds dt H psi (norm up to m dt (1 + 1.25 links) + m dt U) with a few
    # roundings for each link, and keeps the state's own rounding in a second word
    hd = m * dt * (1.0 + 1.25 * links + U)
    tol = steps * ((links + 12) * hd + 1) * 2.0 ** -24
    for r in range(R):
        H1 = np.diag(eps[r])
        for (a, b), j in zip(edges, J[r]):
            H1[a, b] -= j
            H1[b, a] -= j
        ref = v[r].astype(np.complex128).reshape((N,) * m)
        for _ in range(steps):
            ref = ref - 1j * dt * _apply(ref, H1, U, m)
        assert np.linalg.norm(got[:, r] - ref.reshape(-1)) <= tol
