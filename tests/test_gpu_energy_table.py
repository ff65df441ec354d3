"""The FP32 environment pair energy, one pair per replica: r, 1 / r and 1 / r^2 from the
corrected reciprocal root and erfc from its table, from short contacts to the cutoff, for
beta r_c up to the 3.6 that FP32 contexts accept.

Bounds in units of u = 2^-24 of the term, from binary32 inputs: charges and their product
3 u, 1 / r 4 u, the table's value 3 u, products 2 u; r and the table's argument are off by
4 u together, which erfc(beta r) multiplies by at most 2 (beta r)^2 + 1. Lennard-Jones:
parameters 4 u, (sigma / r)^12 twelve times r's 3 u and 6 roundings.
"""
import numpy as np
import pytest

import abfe_synth as S

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def _pair(r, rng, box=3.0):
    d = rng.normal(size=3)
    a = rng.uniform(0.4, box - 0.4, 3)
    pos = S.f32(np.mod(np.stack([a, a + d / np.linalg.norm(d) * r, a + 1.4]), box))
    return S.System("pair", S.f32(np.full(3, box)), pos, np.zeros((3, 3)), np.full(3, 12.0),
                    S.f32(np.array([0.7, -0.5, 0.0])), S.f32(np.array([0.32, 0.28, 0.3])),
                    S.f32(np.array([0.6, 0.4, 0.0])), np.array([0, 0, 1], np.uint8), np.zeros((0, 2), np.int32),
                    np.zeros((0, 2), np.int32), np.zeros(0), np.zeros(0))


@pytest.mark.parametrize("cutoff,beta", [(0.6, 0.5), (0.6, 6.0), (1.0, 3.12), (1.2, 3.0), (1.4, 1.0)])
def test_one_pair(cutoff, beta):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from math import erfc

    import paper_2603_22274_gb300 as G
    rng = np.random.default_rng(int(100 * cutoff + beta))
    m = 48
    systems = [_pair(r, rng) for r in np.linspace(0.12, cutoff - 1e-4, m)]
    P = S.params_for(cutoff, beta)
    w = S.Workload("pairs", systems, np.arange(m, dtype=np.int32), [S.schedule_k12()], np.zeros(m, np.int32),
                   np.zeros(m, np.int32), P)
    eng = G.engine_for_workload(w, precision=0)
    _, E, _ = eng.compute()
    X = eng.positions()
    for i, s in enumerate(systems):
        x = X[eng.offsets[i]:eng.offsets[i + 1]]
        d = x[0] - x[1]
        d -= s.box * np.round(d / s.box)
        r = np.sqrt(d @ d)
        c = P["coulomb_k"] * s.charge[0] * s.charge[1] * erfc(beta * r) / r
        a = (0.5 * (s.sigma[0] + s.sigma[1]) / r) ** 6
        e4 = 4.0 * np.sqrt(s.epsilon[0] * s.epsilon[1])
        assert abs(E[i, 1] - c) <= (12 + 4 * (2 * (beta * r) ** 2 + 1)) * U * abs(c) + 1e-9, (r, E[i, 1], c)
        assert abs(E[i, 0] - e4 * (a * a - a)) <= 46 * U * e4 * (a * a + a) + 1e-9, (r, E[i, 0])
    eng.close()


@pytest.mark.parametrize("cutoff,beta", [(0.9, 3.47), (1.4, 1.0), (1.4, 6.4)])
def test_one_pair_fp64(cutoff, beta):
    """FP64 pairs up to beta r = 9 (the table ends at 8): energies and forces are stored in
    steps of 2^-32, so 1e-9 absolutely; 1e-13 of the term covers 20 roundings at 2 x^2 = 150.
    The pairs lie inside the box: in a gas this thin one cluster spans it, and an image's
    shift relative to the cluster's first atom is rounded to binary32."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from math import erfc, exp, pi

    import paper_2603_22274_gb300 as G
    rng = np.random.default_rng(int(100 * cutoff + beta))
    m = 48
    systems = [_pair(r, rng) for r in np.linspace(0.12, cutoff - 1e-4, m)]
    for s, r in zip(systems, np.linspace(0.12, cutoff - 1e-4, m)):
        d = rng.normal(size=3)
        s.pos[:2] = S.f32(np.stack([np.full(3, 1.5), 1.5 + d / np.linalg.norm(d) * r]))
    P = S.params_for(cutoff, beta)
    w = S.Workload("pairs", systems, np.arange(m, dtype=np.int32), [S.schedule_k12()], np.zeros(m, np.int32),
                   np.zeros(m, np.int32), P)
    eng = G.engine_for_workload(w, precision=1)
    F, E, _ = eng.compute()
    X = eng.positions()
    for i, s in enumerate(systems):
        o = eng.offsets[i]
        d = X[o] - X[o + 1]
        d -= s.box * np.round(d / s.box)
        r = np.sqrt(d @ d)
        qq = P["coulomb_k"] * s.charge[0] * s.charge[1]
        c = qq * erfc(beta * r) / r
        a = (0.5 * (s.sigma[0] + s.sigma[1]) / r) ** 6
        e4 = 4.0 * np.sqrt(s.epsilon[0] * s.epsilon[1])
        f = ((c + qq * 2.0 * beta / np.sqrt(pi) * exp(-(beta * r) ** 2) + e4 * (12.0 * a * a - 6.0 * a)) / r) * d / r
        big = (abs(c) + e4 * (12.0 * a * a + 6.0 * a)) / r
        assert abs(E[i, 1] - c) <= 1e-13 * abs(c) + 1e-9, (r, E[i, 1], c)
        assert abs(E[i, 0] - e4 * (a * a - a)) <= 1e-13 * e4 * (a * a + a) + 1e-9, (r, E[i, 0])
        assert np.all(np.abs(F[o] - f) <= 1e-13 * big + 1e-9) and np.all(np.abs(F[o + 1] + f) <= 1e-13 * big + 1e-9)
    eng.close()
