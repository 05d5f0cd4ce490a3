"""The streaming form where its stage ring wraps and a CTA takes several tiles, and on
the sides of its boundary search, for every storage type and number of harmonics.

Int16 values are small integers, so the same scene in float is the same numbers and has
to give the same bits, and so have columns of it run alone, a tile per CTA, as the
tests against the oracle run them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bfm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_01751_gb300 as bfm
    bfm.load()
    return bfm


def scene(m, N, n, seed):
    """int16 [N][m]: season, noise, steps, clouds."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    t = torch.arange(N, device="cuda", dtype=torch.float32)[:, None]
    Y = torch.empty((N, m), dtype=torch.int16, device="cuda")
    for a in range(0, m, 1 << 18):
        b = min(m, a + (1 << 18))
        y = 5000 + 2000 * torch.sin(2 * np.pi * t / 23.0) + 400 * torch.randn(N, b - a, generator=g, device="cuda")
        y[(n + N) // 2:, ::7] -= 4000
        y = y.round()
        y[torch.rand(N, b - a, generator=g, device="cuda") < 0.3] = -32768
        Y[:, a:b] = y.to(torch.int16)
    return Y


def same(a, b):
    for key in a:
        x, y = a[key], b[key].contiguous()
        if x.dtype == torch.float32:
            ok = (x.view(torch.int32) == y.view(torch.int32)) | (torch.isnan(x) & torch.isnan(y))
        else:
            ok = x == y
        assert ok.all(), (key, int((~ok).sum()))


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("k,N,n,h,lam", [
    (1, 60, 30, 0.25, 1.7),   # six int16 stages
    (2, 61, 29, 0.5, 1.7),
    (3, 64, 40, 0.1, 1.7),
    (3, 90, 20, 0.5, 0.8),    # positions beyond e n_p, many crossings
    (1, 130, 17, 0.25, 2.5),
    (3, 600, 530, 0.02, 1.7),  # one CTA per SM, a ring shorter than the sums kept in it
    (3, 580, 520, 0.05, 1.7),  # and a longer one
])
def test_several_tiles(bfm, k, N, n, h, lam, masked):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m = 256 * 2 * sms * 3 + 264  # three tiles per CTA of two per SM and a ragged fourth
    Y = scene(m, N, n, N + k)
    F = torch.where(Y == -32768, float("nan"), Y.float())
    bits = None
    if masked:
        g = torch.Generator(device="cuda")
        g.manual_seed(k)
        words = torch.randint(-2 ** 31, 2 ** 31, (2, N, (m + 31) // 32), generator=g, device="cuda", dtype=torch.int64)
        bits = (words[0] | words[1]).to(torch.int32)
    dates = np.arange(1.0, N + 1)
    d = bfm.Design(dates, k, 23.0)

    def run(y, mk):
        out = bfm.monitor(d, y, n_hist=n, h_frac=h, lam=lam, mask_bits=mk, algo=bfm.BFM_ALGO_STREAM, max_mosum=True)
        torch.cuda.synchronize()
        assert bfm.bfm_device_errors() == 0
        return out

    full = run(Y, bits)
    same(full, run(F, bits))
    # the first and the last 2048 pixels (32-pixel aligned, for the mask words)
    for a in (0, (m - 2048) // 32 * 32):
        part, mk = F[:, a:a + 2048].contiguous(), None if bits is None else bits[:, a // 32:(a + 2048) // 32].contiguous()
        same(run(part, mk), {key: v[..., a:a + 2048] for key, v in full.items()})


@pytest.mark.parametrize("k", [1, 2, 3])
def test_long_rows(bfm, k):
    """Int16 rows beyond 4 MB."""
    N, n, m = 48, 26, 2 ** 21 + 8
    Y = scene(m, N, n, k)
    d = bfm.Design(np.arange(1.0, N + 1), k, 23.0)
    full = bfm.monitor(d, Y, n_hist=n, h_frac=0.25, lam=1.7, algo=bfm.BFM_ALGO_STREAM)
    for a in (0, m - 2056):
        got = bfm.monitor(d, Y[:, a:a + 2056].float().masked_fill(Y[:, a:a + 2056] == -32768, float("nan")).contiguous(),
                          n_hist=n, h_frac=0.25, lam=1.7, algo=bfm.BFM_ALGO_STREAM)
        same(got, {key: v[..., a:a + 2056] for key, v in full.items()})
    assert bfm.bfm_device_errors() == 0
