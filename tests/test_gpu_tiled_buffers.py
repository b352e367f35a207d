"""The register tiles at the edges of what their loads and their choice of
depth depend on: buffers that start off a 16-byte boundary (8-byte copies
instead of 16-byte ones), lattice sides around whole numbers of tiles, and
every depth the default picks."""
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
    psi = torch.zeros(n + shift, dtype=torch.complex64, device="cuda")[shift:]
    ctqw.ctqw_init_state(h, psi, ctqw.initial_sites(w, h), w.dtype)
    ws = torch.empty(3 * 8 * n + 8 * shift, dtype=torch.uint8, device="cuda")[8 * shift:]
    ctqw.ctqw_propagate_taylor(h, psi, w.dtype, w.dt, w.K, w.n_steps, flags=flags, workspace=ws)
    ctqw.ctqw_check_status(h)
    out = psi.cpu().numpy()
    h.close()
    return out


@pytest.mark.parametrize("N,periodic", [(96, False), (100, True), (97, True), (320, False)])
@pytest.mark.parametrize("K", [4, 7, 8, 16])
def test_unaligned_buffers_give_the_same_bits(ctqw, N, periodic, K):
    # the same arithmetic on the same values: equal to the last bit
    w = cw.get("bosons_n256_u2").with_(N=N, R=3, periodic=periodic, K=K, n_steps=5, obs_every=0,
                                       sites=(N // 2 - 1, N // 2))
    assert np.array_equal(_run(ctqw, w), _run(ctqw, w, shift=1))


@pytest.mark.parametrize("N", [2, 17, 47, 48, 49, 56, 57, 96, 97, 112, 113, 161])
@pytest.mark.parametrize("K", [1, 3, 5, 8, 13, 16])
def test_default_depth_against_per_term(ctqw, N, K):
    # both sides: FP32 Horner stages and a compensated update.  A step's
    # increment (norm <= 0.3) carries a few roundings of 2^-24 per stage, six
    # steps below 6 * 0.3 * 16 * 2^-24 = 1.7e-6 in any amplitude
    w = cw.get("ragged_n128_1024").with_(R=4, ragged_sizes=(N,), sites=(-1, 0), K=K, n_steps=6, obs_every=0)
    a, b = _run(ctqw, w), _run(ctqw, w, flags=ctqw.FLAG_PLAIN)
    assert np.max(np.abs(a - b)) <= 1.7e-6
