"""MBAR iterations at the edges of the device kernel's tiles: one state, state
counts on both sides of its tile widths (256 down to 16 samples) and of its 256
threads, sample counts below one tile, and states without samples.

Both sides apply the same map five times from f = 0 (no convergence test hits), so
f agrees to the rounding of sums of at most N positive FP64 terms, N eps ~ 2e-13 for
the 1,800 samples here, carried through five iterations: tolerance 1e-11.
"""
import numpy as np
import pytest

from oracle.mbar import mbar as mbar_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,per", [(1, 40), (2, 15), (3, 600), (49, 17), (50, 36), (100, 9),
                                   (128, 9), (129, 11), (194, 8), (256, 3), (257, 3), (387, 3),
                                   (388, 3), (1024, 1)])
def test_five_iterations_match_oracle(K, per):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_22274_gb300 as G
    rng = np.random.default_rng(K)
    N_k = np.full(K, per) + (np.arange(K) % 3)
    if K > 2:
        N_k[K // 2] = 0
    ks = 1.1 ** (np.arange(K) % 40)
    x = np.concatenate([rng.normal(0.0, 1.0 / np.sqrt(k), n) for k, n in zip(ks, N_k)])
    u = 0.5 * ks[:, None] * x[None, :] ** 2 + rng.uniform(0.0, 3.0, K)[:, None]
    ref, it_ref = mbar_oracle(u, N_k, tol=1e-300, max_iter=5)   # (one state: exact at once)
    f, it = G.mbar(torch.tensor(u, device="cuda"), N_k, tol=1e-300, max_iter=5)
    assert it == it_ref
    assert np.abs(f - ref).max() <= 1e-11, np.abs(f - ref).max()
