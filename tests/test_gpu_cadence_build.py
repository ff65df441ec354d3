"""The cadence tuner times the build that a forced rebuild and the step graph run: the
ligand clusters' lists on a stream beside the environment's (read from a device trace)."""
import json

import numpy as np
import pytest

import abfe_synth as S

pytestmark = pytest.mark.gpu
SKINS = 5   # candidate outer skins, each built twice (warm, then timed)


def test_tuner_builds_ligand_lists_beside_the_environments(tmp_path):
    import torch
    from torch.profiler import ProfilerActivity, profile
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    s = S.complex_leg(77, n_atoms=6000, core_diameter=2.0, n_lig=30)
    w = S.Workload("mid-6000", [s], np.zeros(1, np.int32), [S.schedule_k42()], np.zeros(1, np.int32),
                   np.array([20], np.int32), S.params_for(1.0, 3.12))
    eng = G.engine_for_workload(w)
    with profile(activities=[ProfilerActivity.CUDA]):   # (a first trace can miss launches)
        eng.compute()
        torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        eng.autotune_cadence(dt=0.0005, gamma=5.0, seed=3, n_steps=8)
        torch.cuda.synchronize()
    path = str(tmp_path / "trace.json")
    prof.export_chrome_trace(path)
    eng.close()
    with open(path) as f:
        ev = [e for e in json.load(f)["traceEvents"] if e.get("cat") == "kernel"]
    ev.sort(key=lambda e: e["ts"])
    streams = {k: [e["args"]["stream"] for e in ev if k in e["name"]]
               for k in ("k_build_list_env", "k_build_list_lig", "k_build_prefix")}
    assert len(streams["k_build_list_lig"]) == len(streams["k_build_prefix"]) > 0
    main = set(streams["k_build_prefix"])
    beside = sum(x not in main for x in streams["k_build_list_lig"])
    assert beside >= 2 * SKINS, (beside, len(streams["k_build_list_lig"]))
