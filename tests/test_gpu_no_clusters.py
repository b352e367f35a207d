"""A handle whose device holds no cluster of the fused kernel: its calls run as
those of sizes that kernel does not take, with the results of the per-term path."""
import numpy as np
import pytest

import ctqw_workloads as cw

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctqw():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1612_00746_gb300 import build, ctqw as c

    build.build()
    c.load()
    return c


def test_null_handle():
    from paper_1612_00746_gb300 import build, ctqw as c

    build.build()
    assert c.load().ctqw_inject_no_clusters(None) == c.CTQW_EINVAL


@pytest.mark.gpu
@pytest.mark.parametrize("call", ["taylor", "rk4", "switching"])
@pytest.mark.parametrize("N,periodic", [(100, False), (256, False), (64, True)])
def test_calls_without_clusters(ctqw, N, periodic, call):
    w = cw.get("bosons_n256_u2").with_(N=N, R=3, K=7, n_steps=5, obs_every=2, periodic=periodic,
                                       sites=(N // 2 - 1, N // 2))
    out = []
    for flags in (0, ctqw.FLAG_PLAIN):
        h = ctqw.build_for_workload(w)
        if flags == 0:
            ctqw.ctqw_inject_no_clusters(h)
            assert ctqw.ctqw_fused_split(h, w.K) == 0
        psi = h.new_state(cw.C64)
        ctqw.ctqw_init_state(h, psi, ctqw.initial_sites(w, h), cw.C64)
        P, nr, en = ctqw._outputs(h, h.n_obs(w.n_steps, 2), True, True, True, "cuda")
        ws = torch.empty(3 * 8 * h.total_amplitudes, dtype=torch.uint8, device="cuda")
        if call == "taylor":
            ctqw.ctqw_propagate_taylor(h, psi, cw.C64, w.dt, w.K, w.n_steps, 2, P, nr, en, flags, ws)
        elif call == "rk4":
            ctqw.ctqw_propagate_rk4(h, psi, cw.C64, w.dt, w.n_steps, 2, P, nr, en, flags,
                                    h.workspace(cw.C64, ctqw.RK4, flags))
        else:
            ctqw.ctqw_propagate_taylor_switching(h, psi, cw.C64, w.dt, w.K, w.n_steps, 2, P, nr, en, 3, 0.2, flags, ws)
        ctqw.ctqw_check_status(h)
        out.append([t.cpu().numpy() for t in (psi, P, nr, en)])
        h.close()
    # FP32 stages on both sides: a step's increment (norm <= 0.3) carries a few
    # roundings of 2^-24 per stage, five steps of 7 stages below
    # 5 x 0.3 x 8 x 7 x 2^-24 = 5e-6 in any amplitude; RK4's plain state update
    # adds half an ulp a step
    for a, b in zip(out[0], out[1]):
        assert np.max(np.abs(a - b)) <= 9 * 2 * 5e-6
