"""Calls that reach the same arithmetic by another route give the same bits: an
explicit mask against missing values, pixel pairs against the one-pixel kernel
(which a mask selects), the layouts TMA cannot take against those it can."""
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


def scene(m, N, n, dtype, missing, seed):
    """Y [N][m] with breaks, clouds, and pixels without data, without history, constant."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    t = torch.arange(N, device="cuda", dtype=torch.float32)[:, None]
    Y = 0.5 + 0.2 * torch.sin(2 * np.pi * t / 23.0) + 0.04 * torch.randn(N, m, generator=g, device="cuda")
    Y[(n + N) // 2:, ::7] -= 0.4
    gone = torch.rand(N, m, generator=g, device="cuda") < missing
    if missing:
        gone[:, 3] = True
        gone[:n, m // 2] = True
        gone[n:, m // 3] = True
    Y[:, 5] = 0.25
    if dtype == torch.int16:
        Y = (Y * 1e4).round().to(torch.int16)
        Y[gone] = -32768
    else:
        Y[gone] = float("nan")
    return Y.contiguous()


def words(bits):
    N, m = bits.shape
    w = -(-m // 32)
    b = torch.zeros((N, w * 32), dtype=torch.int64, device="cuda")
    b[:, :m] = bits
    v = (b.reshape(N, w, 32) << torch.arange(32, device="cuda")).sum(-1)
    return torch.where(v >= 2 ** 31, v - 2 ** 32, v).to(torch.int32).contiguous()


def run(bfm, Y, k, n, h, algo, mask=None):
    d = bfm.Design(np.arange(1.0, Y.shape[0] + 1), k, 23.0)
    out = bfm.monitor(d, Y, n_hist=n, h_frac=h, lam=1.7, mask_bits=mask, algo=algo, max_mosum=True)
    torch.cuda.synchronize()
    return out


def same(a, b, m=None):
    for key in a:
        x, y = a[key], b[key][..., :m]
        if x.dtype == torch.float32:
            ok = (x.view(torch.int32) == y.contiguous().view(torch.int32)) | (torch.isnan(x) & torch.isnan(y))
        else:
            ok = x == y
        assert ok.all(), (key, int((~ok).sum()))


@pytest.mark.parametrize("dtype", [torch.float32, torch.int16])
@pytest.mark.parametrize("form", ["HYBRID", "STREAM", "MMA", "SIMT"])
@pytest.mark.parametrize("m,N,n,k,h", [(1000, 120, 71, 3, 0.25), (136, 65, 33, 1, 0.5), (2008, 97, 64, 2, 0.25)])
def test_mask_is_missing(bfm, form, dtype, m, N, n, k, h):
    """Dates whose mask bit is clear are dates whose value is missing."""
    Y = scene(m, N, n, dtype, 0.2, m)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    keep = torch.rand(N, m, generator=g, device="cuda") < 0.8
    Z = Y.clone()
    Z[~keep] = float("nan") if dtype == torch.float32 else -32768
    algo = getattr(bfm, "BFM_ALGO_" + form)
    same(run(bfm, Z, k, n, h, algo), run(bfm, Y, k, n, h, algo, words(keep)))


@pytest.mark.parametrize("dtype", [torch.float32, torch.int16])
@pytest.mark.parametrize("extra,N,n,k,h", [(0, 60, 33, 1, 0.25), (8, 53, 40, 3, 0.25), (504, 48, 24, 2, 1.0),
                                           (8, 17, 9, 1, 0.1)])
def test_pairs(bfm, dtype, extra, N, n, k, h):
    """Complete scenes large enough for pixel pairs, against the one-pixel kernel."""
    m = 512 * torch.cuda.get_device_properties(0).multi_processor_count + extra
    Y = scene(m, N, n, dtype, 0.0, N)
    Y[N - 1, m - 1] = float("nan") if dtype == torch.float32 else -32768  # one incomplete pixel
    ones = words(torch.ones_like(Y, dtype=torch.bool))
    same(run(bfm, Y, k, n, h, bfm.BFM_ALGO_COMPLETE), run(bfm, Y, k, n, h, bfm.BFM_ALGO_COMPLETE, ones))


@pytest.mark.parametrize("dtype", [torch.float32, torch.int16])
@pytest.mark.parametrize("m,N,n,k", [(33, 70, 40, 3), (1001, 300, 150, 2), (31, 45, 20, 1)])
def test_plain_loads(bfm, dtype, m, N, n, k):
    """The CUDA-core form on rows TMA cannot take, against the same pixels in padded rows."""
    Y = scene(-(-m // 32) * 32, N, n, dtype, 0.3, m)
    narrow = Y[:, :m].contiguous()
    same(run(bfm, narrow, k, n, 0.25, bfm.BFM_ALGO_SIMT), run(bfm, Y, k, n, 0.25, bfm.BFM_ALGO_SIMT), m)
