"""Patch medians and MADs at the awkward inputs of an order-statistic search: negative powers, equal
values around the middle ranks, one value everywhere, infinities, a base 4 bytes past an 8-byte
boundary.  The statistics are order statistics of FP32 numbers: exact against numpy in FP32."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0910_1517_gb300 import build, corr
    build.build()
    corr.load()
    return torch, corr


def _patches():
    r = np.random.default_rng(3)
    P = [r.gamma(32.0, size=4096), r.normal(size=4096), np.round(r.normal(size=4096) * 2),
         np.full(4096, 7.5), np.r_[np.full(2048, -1.0), np.full(2048, 3.0)],
         np.r_[np.full(2047, -1e30), np.full(2, 0.0), np.full(2047, 1e-30)], r.gamma(32.0, size=4096)]
    P[-1][:100] = np.inf
    return np.stack([r.permutation(p) for p in P]).astype(np.float32).reshape(-1, 64, 64)


@pytest.mark.parametrize("shift", [0, 1])
def test_patch_order_statistics(env, shift):
    torch, corr = env
    P = _patches()
    n = len(P)
    buf = torch.empty(P.size + shift, dtype=torch.float32, device="cuda")[shift:]
    buf.copy_(torch.from_numpy(P.reshape(-1)))
    x = torch.empty((n, 64, 64), dtype=torch.float16, device="cuda")
    fl = torch.empty((n, 64, 64), dtype=torch.uint8, device="cuda")
    st = torch.empty((n, 2), dtype=torch.float32, device="cuda")
    corr.rfi_patches(buf, n, 64, 64, 5.0, x, fl, st, stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    s = np.sort(P.reshape(n, -1), axis=1)
    med = np.float32(0.5) * (s[:, 2047] + s[:, 2048])
    d = np.sort(np.abs(P.reshape(n, -1) - med[:, None]), axis=1)
    mad = np.float32(0.5) * (d[:, 2047] + d[:, 2048])
    assert np.array_equal(st.cpu().numpy(), np.stack((med, mad), 1))
    sig = (mad / np.float32(0.6745)).astype(np.float32)
    dev = P - med[:, None, None]
    thr = np.float32(5.0) * sig
    # flags: equal except within one rounding of the threshold
    near = np.abs(np.abs(dev) - thr[:, None, None]) <= 1e-6 * thr[:, None, None]
    assert np.array_equal((fl.cpu().numpy() != 0)[~near], (np.abs(dev) > thr[:, None, None])[~near])
    with np.errstate(all="ignore"):
        u = np.where(sig[:, None, None] > 0, dev / sig[:, None, None], 0.0).astype(np.float64)
    z = np.sign(u) * np.log1p(np.abs(u))
    g = x.float().cpu().numpy()
    fin = np.isfinite(z)
    assert np.array_equal(fin, np.isfinite(g)) and np.abs(g - z)[fin].max() <= 2e-3 * max(1.0, np.abs(z[fin]).max())
