"""env_lane_groups against what the FP32 environment kernel evaluates: all eight i atoms
for every lane of every round of 32 rows, so eight groups of 32 pairs per round, at
least enough rounds for all rows, and at most one partly filled round per work item."""
import numpy as np
import pytest

import abfe_synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("system", ["water", "complex"])
@pytest.mark.parametrize("max_entries", [64, 512])
@pytest.mark.parametrize("prune_skin", [0.0, 0.05, 0.1])
def test_eight_groups_per_round(system, max_entries, prune_skin):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    s = S.water_box(21, 3.0) if system == "water" else S.complex_leg(77, n_atoms=6000, core_diameter=2.0, n_lig=30)
    sch = S.schedule_k12()
    w = S.Workload("lanes", [s], np.zeros(1, np.int32), [sch], np.zeros(1, np.int32), np.zeros(1, np.int32),
                   S.params_for(1.0, 3.12))
    eng = G.engine_for_workload(w)
    eng.set_tuning(group=1, max_entries=max_entries, prune_skin=prune_skin, skin=0.2)
    eng.count_pairs()
    st = eng.stats()
    eng.close()
    rows, groups = st["n_rows"] + st["n_xrows"], st["env_lane_groups"]
    assert rows > 0 and groups % 8 == 0
    assert 8 * rows <= 32 * groups <= 8 * (rows + 31 * st["n_items_env"])
