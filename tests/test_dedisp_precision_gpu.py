"""Rounding of the dedisperser's row pass, whose three FFTs keep their points in registers from one to
the next: each runs its passes in the order 16, R2, R3.  With R3, R2, 16 for the second one the same
push was 2.6 % (1024 channels) and 3.7 % (512) further from 64 bits, and 0.1 % from one set of
samples to another; the bounds lie halfway between the two orders' errors."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

F_LO, BW = 1780.0 / 3.0, 100.0 / 3.0


@pytest.mark.parametrize("n_chan,F,O,avg,dm,push,bound", [
    (1024, 4096, 1200, 64, 30.0, 8192, 3.915e-7),        # 3.866e-7; 3.966e-7 in the other order
    (512, 1024, 135, 4, 1.6142, 3614, 3.458e-7),       # 3.396e-7; 3.521e-7
])
def test_row_pass_rounds_as_single_ffts(n_chan, F, O, avg, dm, push, bound):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import dedisp
    from paper_0910_1517_gb300 import build, corr
    build.build()
    corr.load()
    v = (np.random.default_rng(21).standard_normal((push, n_chan, 4)) * 100.0).astype(np.float32)
    d = corr.corr_dd_create(n_chan, F, O, push, dm, F_LO, BW, avg)
    try:
        out = torch.empty((push // (F - O) + 1) * (F - O) * n_chan // avg, dtype=torch.float32, device="cuda")
        n = corr.corr_dd_push_device(d, torch.from_numpy(v).cuda(), out, stream=torch.cuda.current_stream())
        got = out[:n].cpu().numpy().astype(np.float64)
    finally:
        corr.corr_dd_destroy(d)
    vx, vy = v[..., 0].astype(np.float64) + 1j * v[..., 1], v[..., 2].astype(np.float64) + 1j * v[..., 3]
    want = dedisp.coherent_dedisperse(vx, vy, F, O, dm, F_LO, BW, avg)
    assert got.shape == want.shape
    err = np.sqrt(np.mean((got - want) ** 2) / np.mean(want ** 2))
    print(f"{n_chan} channels: {err:.4e}")
    assert err <= bound
