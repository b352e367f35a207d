"""Two calls on one handle at the same time, each with its own state, workspace
and stream: the states they end in have the same bits as when the calls run
one after the other.  Sizes with one CTA a realization and with clusters, with
fewer and with more realizations than run at once."""
import threading

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


def _calls(ctqw, h, w, n):
    """n states of different contents and n workspaces, and a call on each."""
    rng = np.random.default_rng(w.N)
    v = rng.standard_normal((n, h.total_amplitudes)) + 1j * rng.standard_normal((n, h.total_amplitudes))
    psis = [torch.from_numpy((x / np.linalg.norm(x) * np.sqrt(w.R)).astype(np.complex64)).cuda() for x in v]
    spaces = [torch.empty(3 * 8 * h.total_amplitudes, dtype=torch.uint8, device="cuda") for _ in range(n)]

    def call(i, stream, steps, flags=0):
        ctqw.ctqw_propagate_taylor(h, psis[i], cw.C64, w.dt, w.K, steps, 0, None, None, None, flags, spaces[i], stream)

    return psis, call


@pytest.mark.parametrize("N,R", [(64, 40), (64, 700), (100, 60), (100, 400), (200, 20), (256, 7), (256, 40)])
def test_two_streams(ctqw, N, R):
    w = cw.get("bosons_n256_u2").with_(N=N, R=R, sites=(N // 2 - 1, N // 2))
    streams = [torch.cuda.Stream() for _ in range(2)]
    steps = (60, 37)
    out = []
    for overlap in (False, True):
        h = ctqw.build_for_workload(w)
        psis, call = _calls(ctqw, h, w, 2)
        torch.cuda.synchronize()
        for i in range(2):
            for part in range(3):   # several launches a stream
                call(i, streams[i], steps[i])
            if not overlap:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        ctqw.ctqw_check_status(h)
        out.append([p.cpu().numpy() for p in psis])
        h.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("N,R", [(256, 150), (192, 77)])
def test_two_threads_and_the_second_stream(ctqw, N, R):
    # realizations on the handle's second stream, which the calls of both threads fork and join
    w = cw.get("bosons_n256_u2").with_(N=N, R=R, sites=(N // 2 - 1, N // 2))
    streams = [torch.cuda.Stream() for _ in range(2)]
    out = []
    for overlap in (False, True):
        h = ctqw.build_for_workload(w)
        assert ctqw.ctqw_fused_split(h, w.K) > 0 or N < 256
        psis, call = _calls(ctqw, h, w, 2)
        torch.cuda.synchronize()

        def work(i):
            for part in range(20):
                call(i, streams[i], 2 + i)

        threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
        for t in threads:
            t.start()
            if not overlap:
                t.join()
                torch.cuda.synchronize()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        ctqw.ctqw_check_status(h)
        out.append([p.cpu().numpy() for p in psis])
        h.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_a_call_beside_another_calls_capture(ctqw):
    w = cw.get("bosons_n256_u2").with_(R=150)
    h = ctqw.build_for_workload(w)
    assert ctqw.ctqw_fused_split(h, w.K) > 0
    psis, call = _calls(ctqw, h, w, 2)
    start = [p.clone() for p in psis]
    call(0, None, 3)
    call(0, None, 3)
    call(1, None, 3, ctqw.FLAG_ONE_STREAM)
    torch.cuda.synchronize()
    expect = [p.cpu().numpy() for p in psis]
    for p, q in zip(psis, start):
        p.copy_(q)
    captured, other = torch.cuda.Stream(), torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=captured, capture_error_mode="relaxed"):
        call(0, captured, 3)
        call(1, other, 3)   # at once, and not into the graph
        call(0, captured, 3)
    other.synchronize()
    assert np.array_equal(psis[1].cpu().numpy(), expect[1])
    assert torch.equal(psis[0], start[0])
    graph.replay()
    torch.cuda.synchronize()
    ctqw.ctqw_check_status(h)
    assert np.array_equal(psis[0].cpu().numpy(), expect[0])
    h.close()


@pytest.mark.parametrize("outputs", ["PNE", "P", "E", ""])
@pytest.mark.parametrize("N,R,states", [(200, 60, 3), (64, 700, 1), (64, 700, 2), (64, 700, 5), (256, 40, 3), (256, 150, 3)])
def test_where_the_counter_lies(ctqw, N, R, states, outputs):
    # more realizations than clusters: their counter lies in the workspace or
    # in a sample that is written later, whatever these leave room for (launches
    # of several sampling intervals, the last one cut off); against a workspace
    # with room for it behind the states.
    w = cw.get("bosons_n256_u2").with_(N=N, R=R, K=5, sites=(N // 2 - 1, N // 2))
    every, steps = 2, 17
    h = ctqw.build_for_workload(w)
    rng = np.random.default_rng(R)
    v = rng.standard_normal(h.total_amplitudes) + 1j * rng.standard_normal(h.total_amplitudes)
    v = torch.from_numpy((v / np.linalg.norm(v) * np.sqrt(R)).astype(np.complex64)).cuda()
    full = ctqw._outputs(h, h.n_obs(steps, every), True, True, True, "cuda")
    for o in full:
        o.fill_(7.0)
    got = [o if c in outputs else None for c, o in zip("PNE", full)]
    flags = ctqw.FLAG_ONE_STREAM if R != 150 else 0
    psi = v.clone()
    ws = torch.empty(states * 8 * h.total_amplitudes, dtype=torch.uint8, device="cuda")
    ctqw.ctqw_propagate_taylor(h, psi, cw.C64, w.dt, w.K, steps, every, *got, flags, ws)
    ctqw.ctqw_check_status(h)
    ref = v.clone()
    room = torch.empty(3 * 8 * h.total_amplitudes + 16, dtype=torch.uint8, device="cuda")
    again = ctqw._outputs(h, h.n_obs(steps, every), True, True, True, "cuda")
    ctqw.ctqw_propagate_taylor(h, ref, cw.C64, w.dt, w.K, steps, every, *again, flags, room)
    ctqw.ctqw_check_status(h)
    h.close()
    assert torch.equal(psi, ref)
    for a, b in zip(got, again):
        if a is not None:   # the same terms in another order: FP64 sums of order 10
            assert float((a - b).abs().max()) <= 1e-12
