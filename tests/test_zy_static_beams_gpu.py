"""corr_integrate_static writes its beams at any address of a float: results one, two and three
floats past a 16-byte boundary equal the aligned call's, bit by bit, and the floats around them
stay as they were -- where the F-engine shares its last frame blocks among CTAs (few antennas or
frames) and where it does not."""
import numpy as np
import pytest

from synth import make_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [
    (4, 2, 512, 64),        # two frame blocks, shared
    (5, 1, 64, 272),        # two, the last of 16 frames
    (6, 2, 2048, 16),       # two, shared
    (1, 2, 512, 64),        # one antenna: nothing to share
    (4, 1, 4096, 32),       # the 4096-point kernel never shares
])
def test_beams_at_any_float_address(shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0910_1517_gb300 import build, corr
    build.build()
    corr.load()
    n_ant, n_pol, n_fft, n_int = shape
    s = make_config(2, n_ant=n_ant, n_pol=n_pol, n_fft=n_fft, n_int=n_int, seed=8100 + n_fft)
    n = s.x.shape[1]
    xt = torch.zeros((s.n_in, (n + 15) // 16 * 16 + 16), dtype=torch.int8, device="cuda")
    xt[:, :n] = torch.from_numpy(np.ascontiguousarray(s.x)).cuda()
    vis = torch.empty((n_fft // 2, n_ant * (n_ant + 1) // 2, n_pol ** 2, 2), device="cuda")
    size = n_int * n_fft                                 # two beams of n_int x n_fft / 2
    out = []
    for shift in range(4):
        buf = torch.full((size + 8,), -7.0, device="cuda")
        assert buf.data_ptr() % 16 == 0
        beams = buf[shift:shift + size].view(2, n_int, n_fft // 2)
        corr.corr_integrate_static(n_ant, n_pol, n_fft, n_int, xt, vis, beams, s.delay, s.phi0, s.rate, n_avail=n,
                                   stream=torch.cuda.current_stream(), blocking=1)
        b = buf.cpu().numpy()
        assert (b[:shift] == -7.0).all() and (b[shift + size:] == -7.0).all()
        out.append(b[shift:shift + size])
    assert np.isfinite(out[0]).all() and (out[0] >= 0.0).all()
    for v in out[1:]:
        assert np.array_equal(out[0], v)
