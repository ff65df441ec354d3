"""The allocation-free frame call where its one kernel changes shape: fewer atoms
than its blocks, ligand counts off the tile of eight, a cutoff just below half the
box (its queues overflow and are worked off in parts) and one state.

Both sides sum the same pairs in FP64 from the same binary32 inputs; the tolerance
is 1e-9 of the sum of the terms' magnitudes at most (10^5 terms, rounding 1e-16
each), taken as 1e-9 * max|du| + 1e-6 kJ/mol as for the FP64 context.
"""
import numpy as np
import pytest

import abfe_synth as S
import oracle as O

from test_zz_no_alloc import _frame, _no_torsions, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_lig,box,n_atoms,cutoff,K", [(1, 2.2, 100, 0.9, 1), (7, 2.2, 400, 1.09, 5),
                                                        (9, 3.0, 2800, 1.49, 30), (33, 3.0, 2805, 1.2, 30)])
def test_matches_oracle(n_lig, box, n_atoms, cutoff, K):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    s = _no_torsions(S.solvent_leg(16, n_lig=max(n_lig, 3), box=box, n_atoms=n_atoms))
    if n_lig < 3:   # a ligand of one atom: the others become environment
        s.is_ligand[np.where(s.is_ligand)[0][n_lig:]] = 0
    full = S.schedule_solvent_k30()
    sch = S.LambdaSchedule("part", full.lam_r[:K], full.lam_q[:K], full.lam_v[:K])
    P = S.params_for(cutoff, 3.12)
    X = S.f32(np.mod(s.pos, s.box))
    ref = O.ukn_lambda_part(s, P, sch, pos=X)
    out = torch.empty(sch.K, dtype=torch.float64, device="cuda")
    keep = []
    f = _frame(G, s, P, sch, X, keep)
    got = _run(G, f, sch.K, out)
    assert np.abs(got - ref).max() <= 1e-9 * np.abs(ref).max() + 1e-6, np.abs(got - ref).max()
