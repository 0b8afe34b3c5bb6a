"""Blanker statistics where the histogram and the search over it can go wrong: one value only (one
counter takes the whole block), two values on either side of a half-integer median, the ends of
the int8 range, flat noise over all 256 bins, and ragged last blocks of 1 and of 17 samples.
Medians, MADs, thresholds and counts are whole numbers: equal to the oracle's, bit by bit.  The
spectra equal, bit by bit, those of an unblanked handle fed the oracle's blanked samples, with noise
tables shorter than the four samples replaced together as well."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N_ANT, N_POL, N_FFT = 4, 2, 128


def _rows(n, seed):
    rng = np.random.default_rng(seed)
    x = np.empty((N_ANT * N_POL, n), np.int8)
    x[0] = 5
    x[1] = rng.choice([-7, -6], n)
    x[1, :n // 2 * 2:2], x[1, 1:n // 2 * 2:2] = -7, -6                    # the middle pair straddles -6.5
    x[2] = -128
    x[3] = rng.choice([-128, 127], n)
    x[4] = rng.integers(-128, 128, n)
    x[5] = np.where(rng.random(n) < 0.49, 127, -128)
    x[6] = np.clip(np.rint(rng.standard_normal(n) * 0.6), -127, 127)     # MAD 0 or 1
    x[7] = np.clip(np.rint(rng.standard_normal(n) * 60.0), -128, 127)
    return x


@pytest.mark.parametrize("block", [4096, 8192, 32768])
@pytest.mark.parametrize("extra,L", [(1, 64), (17, 2), (0, 1), (17, 4)])
def test_blanker_at_the_edges(orc, block, extra, L):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0910_1517_gb300 import build, corr
    build.build()
    corr.load()
    n_int = block // N_FFT * 2                       # two blocks of frames; the delay adds the ragged one
    n = n_int * N_FFT + extra
    x = _rows(n, 9100 + extra)
    noise = np.random.default_rng(7).standard_normal((N_ANT * N_POL, L)).astype(np.float32)
    delay = np.zeros(N_ANT)
    delay[-1] = extra

    def run(rows, blank):
        h = corr.corr_create(N_ANT, N_POL, N_FFT, n_int)
        corr.corr_set_delays(h, delay, np.zeros(N_ANT), np.zeros(N_ANT))
        if blank:
            corr.corr_set_blanker(h, 3.0, block, noise)
        xt = torch.zeros((N_ANT * N_POL, (n + 15) // 16 * 16 + 16), dtype=torch.int8, device="cuda")
        xt[:, :n] = torch.from_numpy(np.ascontiguousarray(rows)).cuda()
        corr.corr_integrate_device(h, xt, n_avail=n, stream=torch.cuda.current_stream())
        stats = corr.corr_read_blank_stats(h) if blank else None
        spectra = corr.corr_read_spectra(h, 0, N_FFT // 2, n_int)
        corr.corr_destroy(h)
        return stats, spectra

    (stats, used), got = run(x, True)
    xb, want = orc.mad_blank(x, block, 3.0, noise)
    assert used == n and stats.shape == want.shape == (N_ANT * N_POL, (n + block - 1) // block, 4)
    assert np.array_equal(stats, want)
    assert np.array_equal(got, run(xb, False)[1])
