"""Force passes whose list decision runs from a captured graph (from the eighth pass on)
against the direct launches of a context that made fewer passes: same bits, with no
update due, after steps that make prunes and rebuilds due, and after a change of tuning."""
import numpy as np
import pytest

import abfe_synth as S

pytestmark = pytest.mark.gpu


def _run(G, passes, steps, retune):
    w = S.workload_tiny()
    eng = G.engine_for_workload(w, precision=0)
    if retune:
        eng.set_tuning(group=1, max_entries=64, block_threads=128, graph_steps=0, skin=0.0, prune_skin=0.0)
    for _ in range(passes):
        out = eng.compute()
    if steps:
        eng.step(steps, dt=0.001, gamma=5.0, seed=7)
    out = [a.copy() for a in eng.compute()] + [a.copy() for a in eng.compute()]
    out.append(eng.positions())
    eng.close()
    return out


@pytest.mark.parametrize("steps,retune", [(0, False), (1, False), (60, False), (60, True)])
def test_graph_equals_direct(steps, retune):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    a, b = _run(G, 20, steps, retune), _run(G, 1, steps, retune)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def test_tuning_changed_after_capture():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    res = []
    for passes in (20, 1):
        eng = G.engine_for_workload(S.workload_tiny(), precision=0)
        for _ in range(passes):
            eng.compute()
        eng.set_tuning(group=2, max_entries=128, block_threads=256, graph_steps=0, skin=0.0, prune_skin=0.0)
        for _ in range(passes):
            F, E, _ = eng.compute()
        eng.step(10, dt=0.001, gamma=5.0, seed=7)
        F1, E1, _ = eng.compute()
        res.append((F, E, F1, E1))
        eng.close()
    assert all(np.array_equal(x, y) for x, y in zip(*res))
