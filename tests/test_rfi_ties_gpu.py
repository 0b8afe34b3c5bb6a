"""Near ties of the flagger's one-kernel forward pass: networks whose layer 2 or 3 sums, in FP32 and
in order, round to one fp16 number and in 64 bits (or in the tensor core's order) to its neighbour.
Every activation before the layer is 1, so its sums are those of the weights: two large ones of
opposite sign, the first and the last of them in order, and small ones in between, each three
quarters of an FP32 step of the sum they are added to.

At the pixels whose sums are near ties (all but some at the edges, which miss terms) the
probabilities follow the sums in order -- numpy in FP32 -- with two such channels (their near ties fit
the list of a strip) and with every channel (they do not), and they equal those of the layer
kernels, which patches at another alignment take, bit by bit.  Everywhere one run's equal the next
one's.  The other rounding moves them by 2e-5 or more; the head's sums here are exact in FP32, its
sigmoid is good to a few steps of 2^-24: 5e-7."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

B = 3


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0910_1517_gb300 import build, corr
    build.build()
    corr.load()
    return torch, corr


def _sums(w):
    """sum over channels, then taps, of w [channels][9] over a 64 x 64 image of ones: FP32 in order, and FP64."""
    ones = np.zeros((66, 66))
    ones[1:65, 1:65] = 1.0
    a, e = np.zeros((64, 64), np.float32), np.zeros((64, 64))
    for c in range(w.shape[0]):
        for t in range(9):
            term = w[c, t] * ones[t // 3:t // 3 + 64, t % 3:t % 3 + 64]
            a = a + term.astype(np.float32)                   # (the products are exact)
            e = e + term
    return a, e


def _network(layer, n):
    """Parameters, and each pixel's probability from the sums in order and from the exact ones."""
    p = np.zeros(9441, np.float32)
    p[144:160] = 1.0                                          # layer 1: ones
    W2, W3 = p[160:4768].reshape(32, 16, 9), p[4800:9408].reshape(16, 32, 9)
    w = np.zeros((16 if layer == 2 else 32, 9))
    if layer == 2:
        u = 2.0 ** -14                                        # FP32 step of 512 .. 1024
        w[0, 8], w[15, 8] = 512.0, -512.0
        w[1, 0], w[2, 0] = 1.0, 4 * u
        w[3, :5] = 0.75 * u
        W2[:n] = w
        for o in range(16):
            W3[o, o, 4] = W3[o, o + 16, 4] = 1.0
    else:
        u = 2.0 ** -19                                        # FP32 step of 16 .. 32
        p[4768:4800] = 1.0                                    # layer 2: ones
        w[0, 8], w[15, 8] = 16.0, -16.0
        w[1, 0], w[2, 0], w[3, 0] = 1.0, 2.0 ** -11, -4 * u
        w[4, :5] = 0.75 * u
        W3[:n] = w
    p[9424:9440] = 0.0625
    p[9440] = -0.5
    prob = []
    for s in _sums(w):
        a = np.maximum(s, 0).astype(np.float16).astype(np.float64)
        prob.append(1.0 / (1.0 + np.exp(-(n * a / 16 - 0.5))))
    return p, prob


@pytest.mark.parametrize("layer,n", [(2, 2), (2, 32), (3, 2), (3, 16)])
def test_near_ties_are_summed_in_order(env, layer, n):
    torch, corr = env
    p, (want, exact) = _network(layer, n)
    assert np.array_equal(p.astype(np.float16).astype(np.float32), p)
    tie = np.abs(want - exact) > 2e-5                          # the two roundings are told apart
    assert tie.sum() >= 60 * 60
    x = torch.from_numpy(np.random.default_rng(n).normal(size=(B, 64, 64)).astype(np.float16)).cuda()
    shifted = torch.empty(x.numel() + 1, dtype=torch.float16, device="cuda")[1:].view(B, 64, 64)
    shifted.copy_(x)
    net = corr.rfi_create(B)
    try:
        corr.rfi_set_params(net, p)
        out = []
        for v in (x, x, x, shifted):
            prob = torch.full((B, 64, 64), -1.0, device="cuda")
            corr.rfi_infer(net, v, B, prob, stream=torch.cuda.current_stream())
            out.append(prob.cpu().numpy())
    finally:
        corr.rfi_destroy(net)
    err = [np.abs(o - want)[:, tie].max() for o in out]
    print(f"layer {layer}, {n} channels: " + " ".join(f"{e:.1e}" for e in err))
    for o, e in zip(out, err):
        assert e <= 5e-7
        assert np.array_equal(o[:, tie], out[0][:, tie])
    for o in out[1:3]:
        assert np.array_equal(o, out[0])
