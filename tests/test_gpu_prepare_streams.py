"""Force passes whose list decision runs from a captured graph, on streams that the
context does not have to itself: a stream that another thread uses (its work must run
once, whatever the context captures meanwhile), a stream that the caller is capturing
(before and after the context has its graph), and the legacy default stream."""
import threading

import numpy as np
import pytest

import abfe_synth as S

pytestmark = pytest.mark.gpu
LEGACY = 1   # cudaStreamLegacy


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    return G


def _reference(G):
    eng = G.engine_for_workload(S.workload_tiny(), precision=0)
    out = eng.compute()
    eng.close()
    return out


def test_work_of_another_thread_on_the_stream_runs_once(G):
    import torch
    st = torch.cuda.Stream()
    x = torch.zeros(1, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    eng = G.engine_for_workload(S.workload_tiny(), stream=st, precision=0)
    done, sent = threading.Event(), [0]

    def other():
        with torch.cuda.stream(st):
            while not done.is_set():
                x.add_(1.0)
                sent[0] += 1
                if sent[0] % 64 == 0:
                    st.synchronize()   # (bounds the work queued behind the passes)

    t = threading.Thread(target=other)
    t.start()
    try:
        for k in range(24):   # a change of tuning makes the next passes capture again
            eng.set_tuning(prune_skin=0.0, skin=0.05 + 0.01 * (k % 2))
            F, E, _ = eng.compute()
            for _ in range(12):
                F1, E1, _ = eng.compute()
            assert np.array_equal(F, F1) and np.array_equal(E, E1)
    finally:
        done.set()
        t.join()
    torch.cuda.synchronize()
    eng.close()
    assert float(x) == sent[0]


@pytest.mark.parametrize("passes", [8, 14])   # the eighth unforced pass; after the capture
def test_pass_inside_the_callers_capture(G, passes):
    import torch
    w = S.workload_tiny()
    st = torch.cuda.Stream()
    eng = G.engine_for_workload(w, stream=st, precision=0)
    dF = torch.zeros(eng.total_atoms, 3, dtype=torch.float32, device="cuda")
    dE = torch.zeros(eng.R, len(G.ENERGY_NAMES), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for _ in range(passes):
        eng.compute_device(dF, dE)
    torch.cuda.synchronize()
    F, E = dF.cpu(), dE.cpu()
    dF.zero_()
    dE.zero_()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        g.capture_begin(capture_error_mode="thread_local")
        eng.compute_device(dF, dE)
        g.capture_end()
    assert not dE.any()                # captured, not run
    for _ in range(2):
        dF.zero_()
        dE.zero_()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(dF.cpu(), F) and torch.equal(dE.cpu(), E)
    _, E1, _ = eng.compute()
    assert np.array_equal(E1, E.numpy())
    eng.step(5, dt=0.0005, gamma=5.0, seed=3)
    eng.close()


def test_legacy_default_stream(G):
    F, E, _ = _reference(G)
    eng = G.engine_for_workload(S.workload_tiny(), stream=LEGACY, precision=0, torch_alloc=False)
    for _ in range(20):
        F1, E1, _ = eng.compute()
        assert np.array_equal(F, F1) and np.array_equal(E, E1)
    eng.close()
