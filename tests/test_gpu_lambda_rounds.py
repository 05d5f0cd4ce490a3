"""bfm_lambda where a warp takes several paths, on both sides of the ring's limits.

Path r of seed s starts from s A + r B + 1 (the generator that the header documents), so
it is path 0 of the seed s + r B / A (mod 2^64): sampled paths of a long call have to
give the bits of a call of one path, and agree with the oracle as in
test_gpu_lambda.py."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

A, B, M = 0xA0761D6478BD642F, 0xE7037ED1A0B428DB, 1 << 64


@pytest.mark.parametrize("h,T,G,reps", [
    (0.25, 2.0, 65, 60000),   # many rounds; W(1) is the first step of a block
    (0.5, 3.0, 129, 30000),   # and beyond e
    (1.0, 1.1, 3360, 9000),   # the longest ring with two blocks per SM
    (1.0, 1.1, 3600, 20000),  # the lagged steps drawn again, several rounds
    (1.0, 1.1, 3600, 300),    # a ring with one block per SM
    (1.0, 1.2, 1, 5000),      # all statistics 0: the quantile among equal values
    (0.5, 2.0, 2, 3000),
])
def test_rounds(h, T, G, reps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_01751_gb300 as bfm
    seed, alpha = 11, 0.05
    lam, stats = bfm.bfm_lambda(alpha, h, T, G=G, reps=reps, seed=seed, return_stats=True)
    assert lam == np.sort(stats)[int(np.ceil((1 - alpha) * reps)) - 1]
    for r in [0, 1, reps - 1, reps - 2, reps // 2] + list(np.random.default_rng(G).integers(0, reps, 20)):
        s = (seed + int(r) * B * pow(A, -1, M)) % M
        one = bfm.bfm_lambda(alpha, h, T, G=G, reps=1, seed=s, return_stats=True)[1][0]
        ref = oracle.critical_value(alpha, h, T, G=G, reps=1, seed=s, return_stats=True)[1][0]
        assert stats[r] == one, (r, stats[r], one)
        assert abs(one - ref) <= 1e-9 * ref
