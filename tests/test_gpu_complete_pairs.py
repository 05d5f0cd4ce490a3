"""Complete scenes on both sides of the rule that chooses pixel pairs: whole rounds of
tiles, a few tiles more, half a round more and two rounds with a ragged last tile, with
and without the map of the largest |MO|.  The one-pixel kernel (which a mask of ones
selects) gives the same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ext", [False, True])
@pytest.mark.parametrize("dtype", [torch.float32, torch.int16])
@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("rounds,tiles,extra", [(1, 0, 0), (1, 1, -504), (1, 10, 8), (1.5, 1, 8), (2, 2, 264)])
def test_rule(rounds, tiles, extra, k, dtype, ext):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_01751_gb300 as bfm
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m, N, n = 512 * (int(rounds * sms) + tiles) + extra, 50, 30
    g = torch.Generator(device="cuda")
    g.manual_seed(m)
    t = torch.arange(N, device="cuda", dtype=torch.float32)[:, None]
    Y = 0.5 + 0.2 * torch.sin(2 * np.pi * t / 23.0) + 0.04 * torch.randn(N, m, generator=g, device="cuda")
    Y[(n + N) // 2:, ::7] -= 0.4
    if dtype == torch.int16:
        Y = (Y * 1e4).round().to(dtype)
    Y[N - 1, m - 1] = float("nan") if dtype == torch.float32 else -32768
    ones = torch.full((N, (m + 31) // 32), -1, dtype=torch.int32, device="cuda")
    d = bfm.Design(np.arange(1.0, N + 1), k, 23.0)
    a, b = (bfm.monitor(d, Y, n_hist=n, h_frac=0.25, lam=1.7, mask_bits=mask, algo=bfm.BFM_ALGO_COMPLETE, max_mosum=ext)
            for mask in (None, ones))
    for key in a:
        x, y = a[key], b[key]
        if x.dtype == torch.float32:
            ok = (x.view(torch.int32) == y.view(torch.int32)) | (torch.isnan(x) & torch.isnan(y))
        else:
            ok = x == y
        assert ok.all(), (key, int((~ok).sum()))
    assert (a["status"] == 0).sum() == m - 1 and a["status"][m - 1] == bfm.BFM_PX_INCOMPLETE
