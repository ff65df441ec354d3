"""List updates inside the captured list decision of a force pass: its two conditional
bodies (prune; rebuild and prune). After steps nothing is due, since every step updates
the lists at its own positions, and new positions force the direct launches. An update is
due without being forced after a checkpoint of a context with wider skins is loaded: the
lists are rebuilt at the saved build and prune positions with this context's skins, and
the atoms then lie beyond half of them. Against a context that made too few passes for
the capture: the counters rise alike, and forces, energies, pair counts and the steps
that follow have the same bits."""
import dataclasses

import numpy as np
import pytest

import abfe_synth as S
from test_gpu_exchange import _two_groups

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    return G


def _workload(kind):
    if kind == "exchange":
        return _two_groups(seed=4)
    w = S.workload_tiny()
    if kind == "pme":
        w = dataclasses.replace(w, params=dict(w.params, pme_order=4, pme_spacing=0.12))
    return w


def _engine(G, kind, skin, prune_skin):
    eng = G.engine_for_workload(_workload(kind), precision=1 if kind == "fp64" else 0)
    eng.set_tuning(skin=skin, prune_skin=prune_skin)
    if kind == "exchange":
        eng.set_exchange(1000, seed=5)
    return eng


def _load_and_pass(G, kind, path, skin, prune_skin, passes):
    eng = _engine(G, kind, skin, prune_skin)
    for _ in range(passes):
        eng.compute()
    eng.load_checkpoint(path)
    s0 = eng.stats()
    out = list(eng.compute())
    s1 = eng.stats()
    up = tuple(s1[k] - s0[k] for k in ("n_prunes", "n_rebuilds", "n_window_prunes", "n_window_rebuilds"))
    out += [eng.positions(), np.array(eng.count_pairs()), np.array(up)]
    out += [np.array(a) for a in eng.eval_ukn()]
    eng.step(5, dt=0.0005, gamma=5.0, seed=9)
    out += list(eng.compute()) + [eng.positions(), eng.velocities()]
    eng.close()
    return up, out


@pytest.mark.parametrize("kind", ["fp32", "fp64", "pme", "exchange"])
@pytest.mark.parametrize("skin,prune_skin,rebuilds", [(0.3, 0.004, 0), (0.006, 0.004, 1)])
def test_update_due_in_a_captured_pass(G, kind, skin, prune_skin, rebuilds, tmp_path):
    path = str(tmp_path / "c.bin")
    a = _engine(G, kind, 0.3, 0.15)
    a.compute()
    s0 = a.stats()
    a.step(10, dt=0.0001, gamma=5.0, seed=3)
    s1 = a.stats()
    assert s1["n_prunes"] == s0["n_prunes"] and s1["n_rebuilds"] == s0["n_rebuilds"]
    a.save_checkpoint(path)
    a.close()
    up, x = _load_and_pass(G, kind, path, skin, prune_skin, 20)
    ref_up, y = _load_and_pass(G, kind, path, skin, prune_skin, 1)
    assert up == ref_up and up[0] == 1 and up[1] == rebuilds
    for p, q in zip(x, y):
        assert np.array_equal(p, q)
