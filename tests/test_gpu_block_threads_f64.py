"""The tuning's block size in FP64 contexts: the environment kernel launches blocks of
that size (read from a device trace), and results have the same bits at every size."""
import json

import numpy as np
import pytest

import abfe_synth as S

pytestmark = pytest.mark.gpu


def _block_of(path, kernel):
    with open(path) as f:
        ev = json.load(f)["traceEvents"]
    b = [e["args"]["block"] for e in ev if e.get("cat") == "kernel" and kernel in e["name"]]
    assert b, "kernel not in the trace"
    return {tuple(x) for x in b}


@pytest.mark.parametrize("threads", [64, 96, 128, 256])
def test_block_size_takes_effect(threads, tmp_path):
    import torch
    from torch.profiler import ProfilerActivity, profile
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    eng = G.engine_for_workload(S.workload_tiny(), precision=1)
    ref = eng.compute()
    eng.set_tuning(block_threads=threads)
    for _ in range(2):   # (a process's first trace can miss its first launches)
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            out = eng.compute()
            torch.cuda.synchronize()
    path = str(tmp_path / "trace.json")
    prof.export_chrome_trace(path)
    eng.close()
    for a, b in zip(ref, out):
        assert np.array_equal(a, b)
    assert _block_of(path, "k_env_rows_f64") == {(threads, 1, 1)}
