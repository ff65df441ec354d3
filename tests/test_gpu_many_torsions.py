"""Torsions around the block size of the bonded kernel (96 a block): a system of few
torsions beside one of n, the n being copies of the few with their force constants
shared out, so that energies, forces and dU/dlambda are those of the few.

FP64 contexts; a torsion's forces and a block's energies are rounded to 2^-32 once each:
at most 4 x 400 x 2^-33 = 2e-7 kJ/mol/nm on an atom and less in an energy; tolerance 1e-6.
The launch has blocks for all torsions (read from a device trace)."""
import copy
import json

import numpy as np
import pytest

import abfe_synth as S
from paper_2603_22274_gb300 import ENERGY_NAMES

pytestmark = pytest.mark.gpu
E_TORS = ENERGY_NAMES.index("torsion")


def _with_torsions(s, n):
    t = copy.deepcopy(s)
    m = len(s.torsions)
    of = np.arange(n) % m
    share = np.bincount(of, minlength=m)[of]
    t.torsions, t.torsion_n = s.torsions[of], s.torsion_n[of]
    t.torsion_k, t.torsion_phi0 = s.torsion_k[of] / share, s.torsion_phi0[of]
    return t


@pytest.mark.parametrize("n", [95, 96, 97, 192, 193, 400])
def test_copies_equal_the_few(n, tmp_path):
    import torch
    from torch.profiler import ProfilerActivity, profile
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    base = S.solvent_leg(11, n_lig=40, box=3.5)
    assert 0 < len(base.torsions) < 95
    sch = S.schedule_k42()
    st = np.array([5, 5, 20, 20], np.int32)
    w = S.Workload("tors", [base, _with_torsions(base, n)], np.array([0, 1, 0, 1], np.int32), [sch],
                   np.zeros(4, np.int32), st, S.params_for(1.0, 3.12))
    eng = G.engine_for_workload(w, precision=1)
    for _ in range(2):   # (a process's first trace can miss its first launches)
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            F, E, D = eng.compute()
            torch.cuda.synchronize()
    path = str(tmp_path / "trace.json")
    prof.export_chrome_trace(path)
    off = eng.offsets
    eng.close()
    assert abs(E[0, E_TORS]) > 1e-3
    for a, b in ((0, 1), (2, 3)):
        assert np.abs(E[a] - E[b]).max() <= 1e-6 and np.abs(D[a] - D[b]).max() <= 1e-6
        assert np.abs(F[off[a]:off[a + 1]] - F[off[b]:off[b + 1]]).max() <= 1e-6
    with open(path) as f:
        ev = json.load(f)["traceEvents"]
    grids = [e["args"]["grid"] for e in ev if e.get("cat") == "kernel" and "k_restraints" in e["name"]]
    assert grids and all(g[0] == 4 and g[1] == -(-n // 96) for g in grids)
