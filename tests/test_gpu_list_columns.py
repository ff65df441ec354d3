"""Cluster lists from columns on both sides of the sort's ranked sizes (128, 256 and
512 atoms), from empty and nearly empty columns, and in a box so low that the search
takes several z images: every pair in the cutoff is found, per atom, as by brute force.

Pairs whose distance lies within 1e-5 nm of the cutoff may go either way: coordinates
of at most 44 nm and their differences across the box are binary32, to 4e-6 nm.
"""
import numpy as np
import pytest

import abfe_synth as S
import oracle as O

pytestmark = pytest.mark.gpu

CUTOFF = 1.0


def _gas(rng, sizes, lz, box=2.4):
    """Four columns of 1.2 nm (density 8 per nm^3) holding `sizes` atoms, two ligand atoms."""
    parts = []
    for c, n in enumerate(sizes):
        p = rng.uniform(0.0, 1.0, (n, 3)) * [0.498 * box, 0.498 * box, 0.999 * lz] + 1e-3
        p[:, 0] += 0.5 * box * (c // 2)
        p[:, 1] += 0.5 * box * (c % 2)
        parts.append(p)
    pos = S.f32(np.concatenate(parts + [rng.uniform(0.1, 1.0, (2, 3)) * [box, box, lz] * 0.9]))
    n = len(pos)
    lig = np.zeros(n, np.uint8)
    lig[-2:] = 1
    return S.System(f"gas-{n}", S.f32(np.array([box, box, lz])), pos, np.zeros((n, 3)), np.full(n, 12.0),
                    np.zeros(n), np.full(n, 0.2), np.full(n, 0.1), lig, np.zeros((0, 2), np.int32),
                    np.zeros((0, 2), np.int32), np.zeros(0), np.zeros(0))


@pytest.mark.parametrize("legs", [[([126, 127, 128, 129], 11.0)], [([254, 255, 256, 257], 22.0)],
                                  [([510, 511, 512, 513], 44.0)], [([40, 0, 1, 5], 2.4)],
                                  [([127, 129, 128, 126], 11.0), ([520, 505, 512, 513], 44.0), ([20, 18, 15, 21], 2.1)]])
def test_pairs_match_brute_force(legs):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    rng = np.random.default_rng(sum(map(sum, (s for s, _ in legs))))
    systems = [_gas(rng, sizes, lz) for sizes, lz in legs]
    m = len(systems)
    w = S.Workload("gas", systems, np.arange(m, dtype=np.int32), [S.schedule_k12()], np.zeros(m, np.int32),
                   np.arange(m, dtype=np.int32), S.params_for(CUTOFF, 3.12))
    eng = G.engine_for_workload(w, precision=0)
    _, got = eng.count_pairs(per_atom=True)
    X = eng.positions()
    for r, s in enumerate(systems):
        a, b = eng.offsets[r], eng.offsets[r + 1]
        ref = O.neighbor_counts(s, CUTOFF, pos=X[a:b])
        lo = O.neighbor_counts(s, CUTOFF - 1e-5, pos=X[a:b])
        hi = O.neighbor_counts(s, CUTOFF + 1e-5, pos=X[a:b])
        assert np.all((got[a:b] >= lo) & (got[a:b] <= hi))
        exact = lo == hi
        assert np.array_equal(got[a:b][exact], ref[exact])
    eng.close()
