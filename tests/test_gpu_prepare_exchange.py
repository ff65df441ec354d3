"""Force passes between steps of a context with in-loop replica exchange: from the
eighth pass on their list decision runs from a captured graph, which has no exchange
node. Against a context that makes too few passes for the capture: same bits, with
exchanges switched on before and after the capture, and for direct and captured steps."""
import numpy as np
import pytest

from test_gpu_exchange import _two_groups

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    return G


def _run(G, extra, on_first, graph_steps):
    eng = G.engine_for_workload(_two_groups(seed=4))
    eng.set_tuning(graph_steps=graph_steps)
    if on_first:
        eng.set_exchange(5, seed=77)
    for _ in range(1 + extra):
        eng.compute()
    if not on_first:
        eng.set_exchange(5, seed=77)
        for _ in range(extra):
            eng.eval_ukn()
    out = []
    for k in range(4):
        eng.step(5, dt=0.0005, gamma=5.0, seed=100 + k)
        out += [np.array(a) for a in eng.eval_ukn()]
        out.append(np.array(eng.replica_states()))
    out += [np.array(a) for a in eng.compute()] + [eng.positions(), eng.velocities()]
    s = eng.stats()
    assert s["n_exchange_attempts"] == 4
    out.append(np.array(s["n_exchange_accepted"]))
    eng.close()
    return out


@pytest.mark.parametrize("graph_steps", [0, 5])
@pytest.mark.parametrize("on_first", [True, False])
def test_passes_between_exchanging_steps(G, on_first, graph_steps):
    a, b = _run(G, 12, on_first, graph_steps), _run(G, 0, on_first, graph_steps)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
