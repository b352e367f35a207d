"""The second stream's share by rounds of tile blocks: none where two CTAs of
the clusters share an SM (the tiles then keep clusters out), and the results of
one stream where the tiles take several rounds."""
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


@pytest.mark.parametrize("N,R,K", [(200, 600, 16), (196, 350, 16), (219, 33, 8), (250, 48, 16)])
def test_none_where_clusters_share_their_sms(ctqw, N, R, K):
    h = ctqw.build_for_workload(cw.get("bosons_n256_u2").with_(N=N, R=R, sites=(N // 2 - 1, N // 2)))
    assert ctqw.ctqw_fused_split(h, K) == 0
    h.close()


@pytest.mark.parametrize("N,R,K", [(240, 130, 5), (255, 90, 8), (192, 140, 16), (161, 200, 12), (218, 140, 4)])
def test_shares_agree_with_one_stream(ctqw, N, R, K):
    w = cw.get("bosons_n256_u2").with_(N=N, R=R, K=K, sites=(N // 2 - 1, N // 2))
    out = []
    for flags in (0, ctqw.FLAG_ONE_STREAM):
        h = ctqw.build_for_workload(w)
        assert 0 <= ctqw.ctqw_fused_split(h, K) < R // 2
        psi = h.new_state(cw.C64)
        ctqw.ctqw_init_state(h, psi, ctqw.initial_sites(w, h), cw.C64)
        P, nr, en = ctqw._outputs(h, h.n_obs(5, 2), True, True, True, "cuda")
        ctqw.ctqw_propagate_taylor(h, psi, cw.C64, w.dt, K, 5, 2, P, nr, en, flags, h.workspace(cw.C64))
        ctqw.ctqw_check_status(h)
        out.append([t.cpu().numpy() for t in (psi, P, nr, en)])
        h.close()
    # FP32 Horner stages and a compensated update on both sides: a step's
    # increment (norm <= 0.3) carries a few roundings of 2^-24 per stage, five
    # steps below 5 x 0.3 x 16 x 2^-24 = 1.5e-6 in any amplitude
    assert np.max(np.abs(out[0][0] - out[1][0])) <= 1.5e-6
    for a, b in zip(out[0][1:], out[1][1:]):   # 2 |psi| |dpsi|; energies times ||H|| <= 9
        assert np.max(np.abs(a - b)) <= 9 * 3e-6
