"""Non-finite coordinates and velocities are refused wherever they stand, the state
stays as it was to the bit, and the next call works."""
import numpy as np
import pytest

import abfe_synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("where", [0, 1000, -1])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_refused_and_unchanged(where, value):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    w = S.workload_tiny()
    eng = G.engine_for_workload(w, precision=0)
    F, E, _ = eng.compute()
    X, V = eng.positions(), eng.velocities()
    for get, put, a in ((eng.positions, eng.set_positions, X), (eng.velocities, eng.set_velocities, V)):
        bad = a.copy()
        bad.reshape(-1)[where] = value
        with pytest.raises(G.AbfeError):
            put(bad)
        assert np.array_equal(get(), a)
    F1, E1, _ = eng.compute()
    assert np.array_equal(F, F1) and np.array_equal(E, E1)
    eng.set_positions(X)
    F2, E2, _ = eng.compute()
    assert np.array_equal(F, F2) and np.array_equal(E, E2)
    eng.close()
