"""Reciprocal-space Ewald at the grids where the device's transforms change shape: planes
of 90 x 90 points no longer fit in shared memory (the transforms go axis by axis); order 5 (eight lanes per atom, on an odd grid);
and boxes with unequal edges. Same oracle and tolerances as the other PME tests.
"""
import numpy as np
import pytest

import abfe_synth as S

from test_gpu_parity import rel_rms
from test_gpu_pme import E_RECIP, E_TOTAL, grid_for, recip_terms, state_ref

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("points,order", [(45, 5), (48, 4), (54, 6), (60, 4), (90, 4)])
@pytest.mark.parametrize("stretch", [1.0, 1.65])
def test_matches_oracle(points, order, stretch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    s = S.solvent_leg(31, n_lig=8, box=2.2)
    s.box = S.f32(s.box * np.array([1.0, 1.0, stretch]))   # (room above the water)
    s.torsions = s.torsions[:0]
    s.torsion_k, s.torsion_n, s.torsion_phi0 = s.torsion_k[:0], s.torsion_n[:0], s.torsion_phi0[:0]
    P = S.params_for(0.9, 3.47)
    P.update(pme_order=order, pme_spacing=float(s.box[0]) / points)
    assert grid_for(s.box, P["pme_spacing"], order)[0] == points
    sch = S.schedule_solvent_k30()
    w = S.Workload("s", [s], np.zeros(1, np.int32), [sch], np.zeros(1, np.int32), np.array([9], np.int32), P)
    eng = G.engine_for_workload(w, precision=0)
    F, E, _ = eng.compute()
    X = eng.positions()
    lam = sch.state(9)
    Eo, Fo, Er, sc = state_ref(s, P, lam, X)
    assert rel_rms(F, Fo) <= 1e-5, rel_rms(F, Fo)
    assert abs(E[0, E_TOTAL] - Eo) <= 1e-6 * sc, (E[0, E_TOTAL], Eo, sc)
    assert abs(E[0, E_RECIP] - Er) <= 1e-6 * sc, (E[0, E_RECIP], Er, sc)
    ks = list(range(0, sch.K, 7))
    got = eng.eval_ukn()[1][0, ks]
    ref = np.array([state_ref(s, P, sch.state(k), X)[0] for k in ks])
    assert np.abs((got - got[0]) - (ref - ref[0])).max() <= 1e-3
    eng.close()
