"""A batch follows settings that are changed on its handles after its graph was captured: power
dumps turned on, made longer, turned off and on again while another allocation takes the place of
the old buffer; averaged beams of other lengths, likewise; polarisation products.  After each change
the batch's dumps, beams and visibilities equal, bit by bit, those of the same integration by a
fresh batch of fresh handles with these settings from the beginning."""
import numpy as np
import pytest

from synth import make_config

pytestmark = pytest.mark.gpu

SUBS = [(4, 2, 512, 256), (3, 1, 4096, 64), (8, 2, 128, 512)]


@pytest.fixture(scope="module")
def env(orc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0910_1517_gb300 import build, corr
    build.build()
    corr.load()
    return torch, corr


def _handle(corr, s):
    h = corr.corr_create(s.n_ant, s.n_pol, s.n_fft, s.n_int)
    corr.corr_set_delays(h, s.delay, s.phi0, s.rate)
    return h


def _read(corr, h, s, dump):
    out = [corr.corr_read_visibilities(h), corr.corr_read_beams(h)]
    return out + ([corr.corr_read_power_host(h, s.n_int // dump)] if dump else [])


def test_batch_follows_settings_changed_after_capture(env):
    torch, corr = env
    st = torch.cuda.current_stream()
    ss, xs = [], []
    for q, (na, npol, nfft, nint) in enumerate(SUBS):
        s = make_config(2, n_ant=na, n_pol=npol, n_fft=nfft, n_int=nint, seed=8300 + q)
        n = s.x.shape[1]
        xt = torch.zeros((s.n_in, (n + 15) // 16 * 16 + 16), dtype=torch.int8, device="cuda")
        xt[:, :n] = torch.from_numpy(np.ascontiguousarray(s.x)).cuda()
        ss.append(s)
        xs.append((xt, n))
    rows, avail = [x for x, _ in xs], [n for _, n in xs]

    def apply(hs, dumps, avgs, pol):
        for h, d, m in zip(hs, dumps, avgs):
            corr.corr_set_mode(h, corr.CORR_FP32, pol, m)
            corr.corr_set_power_dump(h, d)

    def run(b, hs, dumps):
        corr.corr_batch_integrate_device(b, rows, n_avail=avail, stream=st)
        return [_read(corr, h, s, d) for h, s, d in zip(hs, ss, dumps)]

    hs = [_handle(corr, s) for s in ss]
    others = []                                          # handles outside the batch, whose buffers take freed places
    b = corr.corr_batch_create(hs)
    try:
        # (dump lengths, beam averages, polarisation products, off in between)
        steps = [((0, 0, 0), (1, 1, 1), 0, False), ((16, 16, 16), (1, 1, 1), 0, False), ((32, 8, 64), (4, 1, 8), 0, False),
                 ((32, 8, 64), (4, 1, 8), 0, True), ((8, 4, 8), (16, 2, 2), 0, True), ((0, 0, 16), (1, 1, 1), 1, False),
                 ((16, 16, 16), (2, 2, 2), 0, True)]
        for dumps, avgs, pol, off in steps:
            if off:
                before = list(zip(dumps, avgs))
                apply(hs, (0, 0, 0), (1, 1, 1), pol)
                for s, (d, m) in zip(ss, before):
                    o = _handle(corr, s)
                    others.append(o)
                    apply([o], [d], [m], pol)
            apply(hs, dumps, avgs, pol)
            got = run(b, hs, dumps)
            fresh = [_handle(corr, s) for s in ss]
            fb = None
            try:
                apply(fresh, dumps, avgs, pol)
                fb = corr.corr_batch_create(fresh)
                want = run(fb, fresh, dumps)
            finally:
                if fb is not None:
                    corr.corr_batch_destroy(fb)
                for h in fresh:
                    corr.corr_destroy(h)
            for g, w in zip(got, want):
                assert len(g) == len(w)
                for u, v in zip(g, w):
                    assert np.isfinite(u).all() and np.abs(u).max() > 0.0
                    assert u.shape == v.shape and np.array_equal(u, v), (dumps, avgs, pol)
    finally:
        corr.corr_batch_destroy(b)
        for h in hs + others:
            corr.corr_destroy(h)
