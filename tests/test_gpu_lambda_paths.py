"""Path statistics of bfm_lambda where the kernel's blocks of 32 steps and its
ring meet their edges, against the oracle (the same draws; tolerance as in
test_gpu_lambda.py)."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,T,G,reps", [
    (1.0, 1.2, 8000, 40),    # h G beyond the shared-memory ring: the lagged steps drawn again
    (1.0, 1.5, 64, 33),      # the lag reaches W(0); G a multiple of 32
    (0.01, 1.3, 100, 130),   # a lag of one step
    (0.25, 3.5, 37, 5),      # a lag within a block of steps; horizon beyond e
    (1.0, 5.0, 1, 7),        # one step per unit time
    (0.3, 1.0001, 320, 1),   # horizon at G
])
def test_paths(h, T, G, reps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_01751_gb300 as bfm
    lam_g, st_g = bfm.bfm_lambda(0.05, h, T, G=G, reps=reps, seed=11, return_stats=True)
    lam_o, st_o = oracle.critical_value(0.05, h, T, G=G, reps=reps, seed=11, return_stats=True)
    assert (np.abs(st_g - st_o) <= 1e-9 * np.maximum(np.abs(st_o), 1e-300)).all()
    assert abs(lam_g - lam_o) <= 1e-9 * lam_o
