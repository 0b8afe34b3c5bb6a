"""Tensor-core X-engine at the edges of its tiles: 256-row Grams (two items a channel) through both
hand-off layouts, integrations that end inside a stage, inside an accumulation chunk and one step
past it, and row counts around the 128-row item.

FP32 form (CORR_FP32TC): the FP32 visibility bound 1e-5 of sqrt(V_aa V_a'a') against the FP64 oracle
on sampled channels.  int8 form: integer visibilities equal the oracle's integer MAC bit for bit."""
import numpy as np
import pytest

from fxhelp import vis_norm_error
from synth import make_config

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env(orc):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0910_1517_gb300 import build, corr
    build.build()
    corr.load()
    return torch, corr, orc


def _run(env, shape, mode):
    torch, corr, orc = env
    n_ant, n_pol, n_fft, n_int = shape
    s = make_config(2, n_ant=n_ant, n_pol=n_pol, n_fft=n_fft, n_int=n_int, seed=7100 + n_ant + n_fft + n_int)
    n = s.x.shape[1]
    xt = torch.zeros((s.n_in, (n + 15) // 16 * 16 + 16), dtype=torch.int8, device="cuda")
    xt[:, :n] = torch.from_numpy(np.ascontiguousarray(s.x)).cuda()
    h = corr.corr_create(n_ant, n_pol, n_fft, n_int)
    corr.corr_set_delays(h, s.delay, s.phi0, s.rate)
    if mode == corr.CORR_I8:
        corr.corr_set_scales(h, np.full((s.n_in, n_fft // 2), 127.0 / (80.0 * np.sqrt(n_fft / 2)), np.float32))
    corr.corr_set_mode(h, mode, 0, 1)
    corr.corr_integrate_device(h, xt, n_avail=n, stream=torch.cuda.current_stream())
    return s, h


@pytest.mark.parametrize("shape", [
    (64, 2, 4096, 48),      # 256 rows, CUDA-core layout: 32-frame stages, the last one half
    (64, 2, 256, 144),      # 256 rows, channel quads: one step past a chunk
    (33, 2, 128, 80),       # 132 rows: a second item of four rows
    (32, 2, 256, 1040),     # paired items: two chunks and one step
    (32, 2, 4096, 80),      # paired items from the CUDA-core layout
    (31, 2, 64, 528),       # 124 rows, three products
    (3, 1, 128, 144),       # six rows
])
def test_fp32_form_at_tile_edges(env, shape):
    torch, corr, orc = env
    s, h = _run(env, shape, corr.CORR_FP32TC)
    try:
        V = corr.corr_read_visibilities(h).astype(np.complex128)
    finally:
        corr.corr_destroy(h)
    chans = np.unique(np.linspace(0, shape[2] // 2 - 1, 16).astype(np.int32))
    Y = orc.fengine(s.x, s.n_ant, s.n_pol, s.n_fft, s.n_int, s.delay, s.phi0, s.rate, chans=chans)
    e = vis_norm_error(V[chans], orc.xengine(Y, s.n_ant, s.n_pol), s.n_ant, s.n_pol)
    print(f"{shape}: {e:.2e}")
    assert e <= 1e-5


@pytest.mark.parametrize("shape", [
    (64, 2, 256, 1040),     # 256 rows: a chunk and one step
    (33, 2, 128, 80),
    (32, 2, 128, 2064),     # 128 rows: two chunks and one step
    (32, 2, 4096, 80),
    (1, 1, 64, 16),         # one input, one step
])
def test_int8_form_at_tile_edges(env, shape):
    torch, corr, orc = env
    s, h = _run(env, shape, corr.CORR_I8)
    try:
        Vi = corr.corr_read_vis_int(h)
        q, sc = corr.corr_read_requant(h, 0, shape[2] // 2, s.n_int)
    finally:
        corr.corr_destroy(h)
    ref, _ = orc.xint(q, sc.astype(np.float64), s.n_ant, s.n_pol)
    assert np.array_equal(Vi, ref.astype(np.int32))
