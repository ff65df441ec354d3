"""MBAR iterations whose matrix is mostly zeros, for state counts at which a warp's lanes
sum different segments of a tile or none: neighbouring lanes then skip different groups
of samples.

Harmonic wells 3 sigma apart: a sample's weights beyond the fifth neighbour are below
2^-160 and stored as zeros. Both sides apply the same map five times from f = 0; f agrees
to the rounding of sums of at most N positive FP64 terms, N eps ~ 4e-13 for the 1,600
samples here, of logarithms of size up to about 100 (2e-14), carried through five
iterations: tolerance 1e-11.
"""
import numpy as np
import pytest

from oracle.mbar import mbar as mbar_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,per", [(5, 300), (12, 40), (33, 20), (80, 20), (100, 13), (200, 5), (300, 3)])
def test_separate_wells_match_oracle(K, per):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    rng = np.random.default_rng(K)
    N_k = np.full(K, per)
    mu = 3.0 * np.arange(K)
    x = np.concatenate([rng.normal(m, 1.0, n) for m, n in zip(mu, N_k)])
    u = 0.5 * (x[None, :] - mu[:, None]) ** 2 + rng.uniform(0.0, 3.0, K)[:, None]
    ref, it_ref = mbar_oracle(u, N_k, tol=1e-300, max_iter=5)
    f, it = G.mbar(torch.tensor(u, device="cuda"), N_k, tol=1e-300, max_iter=5)
    assert it == it_ref
    assert np.abs(f - ref).max() <= 1e-11, np.abs(f - ref).max()
