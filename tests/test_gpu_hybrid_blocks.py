"""The hybrid form in single calls whose CTAs take several blocks of 256 pixels in both
of their groups, with a ragged last block.  Columns run alone (one block, first group)
give the same bits, a mask those of missing values, and int16 storage those of float
(its values are small integers)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def same(a, b):
    for key in a:
        x, y = a[key], b[key].contiguous()
        if x.dtype == torch.float32:
            ok = (x.view(torch.int32) == y.view(torch.int32)) | (torch.isnan(x) & torch.isnan(y))
        else:
            ok = x == y
        assert ok.all(), (key, int((~ok).sum()))


@pytest.mark.parametrize("k,N,n,h", [(1, 61, 33, 0.25), (2, 80, 48, 0.5), (3, 120, 71, 0.25), (3, 75, 30, 1.0)])
def test_blocks(k, N, n, h):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1807_01751_gb300 as bfm
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m = 256 * 4 * sms + 264  # blocks u to CTA u % SMs and group (u / SMs) % 2: two rounds and two blocks more
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    t = torch.arange(N, device="cuda", dtype=torch.float32)[:, None]
    y = 5000 + 2000 * torch.sin(2 * np.pi * t / 23.0) + 400 * torch.randn(N, m, generator=g, device="cuda")
    y[(n + N) // 2:, ::7] -= 4000
    y = y.round()
    gone = torch.rand(N, m, generator=g, device="cuda") < 0.3
    gone[:, 300::1000] = True
    gone[n:, 700::1000] = True
    keep = torch.rand(N, m, generator=g, device="cuda") < 0.85
    w = (m + 31) // 32
    bits = torch.zeros((N, w * 32), dtype=torch.int64, device="cuda")
    bits[:, :m] = keep
    bits = (bits.reshape(N, w, 32) << torch.arange(32, device="cuda")).sum(-1)
    words = torch.where(bits >= 2 ** 31, bits - 2 ** 32, bits).to(torch.int32).contiguous()
    F = y.masked_fill(gone, float("nan"))
    Y = y.masked_fill(gone, -32768).to(torch.int16)
    Z = F.masked_fill(~keep, float("nan"))
    d = bfm.Design(np.arange(1.0, N + 1), k, 23.0)

    def run(v, mask=None):
        out = bfm.monitor(d, v, n_hist=n, h_frac=h, lam=1.7, mask_bits=mask, algo=bfm.BFM_ALGO_HYBRID, max_mosum=True)
        torch.cuda.synchronize()
        assert bfm.bfm_device_errors() == 0
        return out

    full, masked = run(F), run(F, words)
    same(full, run(Y))
    same(masked, run(Y, words))
    same(masked, run(Z))
    for block in (0, 1, sms, 2 * sms - 1, 2 * sms + 3, 3 * sms, 4 * sms):
        a, b = 256 * block, min(m, 256 * block + 256)
        same(run(F[:, a:b].contiguous()), {key: v[..., a:b] for key, v in full.items()})
        same(run(F[:, a:b].contiguous(), words[:, a // 32:(b + 31) // 32].contiguous()),
             {key: v[..., a:b] for key, v in masked.items()})
    a = 256 * (4 * sms + 1)  # the ragged block: 8 pixels
    same(run(F[:, a:].contiguous()), {key: v[..., a:] for key, v in full.items()})
