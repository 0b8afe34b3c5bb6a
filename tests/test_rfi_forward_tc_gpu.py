"""The FP16 flagger's one-kernel forward pass (16-byte aligned patches) against the layer-by-layer
kernels, which the same call runs on patches at any other alignment: both round every activation to
fp16 from an FP32 sum, so they differ by single fp16 steps of an activation at most (2^-11 relative
each, the 2e-3 the flagger's probabilities are held to against the oracle)."""
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


def _params(seed):
    rng = np.random.default_rng(seed)
    p = np.zeros(9441, np.float32)
    for o, n, fan in ((0, 144, 9), (160, 4608, 144), (4800, 4608, 288), (9424, 16, 16)):
        p[o:o + n] = rng.normal(scale=np.sqrt(2.0 / fan), size=n)
    for o, n in ((144, 16), (4768, 32), (9408, 16), (9440, 1)):
        p[o:o + n] = rng.normal(scale=0.1, size=n)
    return p


@pytest.mark.parametrize("B", [1, 3, 38, 77])          # below, at and past one strip a resident CTA
def test_forward_and_gradients_agree_with_the_layer_kernels(env, B):
    torch, corr = env
    rng = np.random.default_rng(B)
    x = torch.from_numpy(rng.normal(size=(B, 64, 64)).astype(np.float16)).cuda()
    x[0, :, 0] = 6.0                                     # edges that matter
    x[-1, 63, :] = -5.0
    m = torch.from_numpy((rng.random((B, 64, 64)) < 0.1).astype(np.uint8)).cuda()
    shifted = torch.empty(x.numel() + 1, dtype=torch.float16, device="cuda")[1:].view(B, 64, 64)
    shifted.copy_(x)
    assert x.data_ptr() % 16 == 0 and shifted.data_ptr() % 16 == 2
    net = corr.rfi_create(B)
    try:
        corr.rfi_set_params(net, _params(5))
        out = []
        for v in (x, shifted):
            prob = torch.full((B, 64, 64), -1.0, device="cuda")
            corr.rfi_infer(net, v, B, prob, stream=torch.cuda.current_stream())
            loss, grad = corr.rfi_loss_grad(net, v, m, B, stream=torch.cuda.current_stream())
            out.append((prob.cpu().numpy(), loss, grad))
    finally:
        corr.rfi_destroy(net)
    (pa, la, ga), (pb, lb, gb) = out
    print(f"B {B}: prob {np.abs(pa - pb).max():.1e} loss {abs(la - lb) / lb:.1e} grad {np.abs(ga - gb).max() / np.abs(gb).max():.1e}")
    assert np.abs(pa - pb).max() <= 2e-3
    assert abs(la - lb) <= 2e-3 * lb
    assert np.abs(ga - gb).max() <= 1e-2 * np.abs(gb).max()


@pytest.mark.parametrize("value", [0.0, 1.0])
def test_constant_patches(env, value):
    """Patches of one value: every interior activation equal, and all of them near ties at once or none."""
    torch, corr = env
    x = torch.full((2, 64, 64), value, dtype=torch.float16, device="cuda")
    net = corr.rfi_create(2)
    try:
        p = np.zeros(9441, np.float32)                   # layer 2 = 1 + 2^-11 at every inner position: a tie
        p[144:160] = 1.0
        p[160:4768] = 0.0
        p[160 + 4:4768:144] = 1.0
        p[4768:4800] = 2.0 ** -11
        p[9408:9424] = 0.5
        p[9424:9440] = 0.1
        corr.rfi_set_params(net, p)
        prob = torch.empty((2, 64, 64), device="cuda")
        corr.rfi_infer(net, x, 2, prob, stream=torch.cuda.current_stream())
        torch.cuda.synchronize()
    finally:
        corr.rfi_destroy(net)
    s = 16 * 0.5 * float(np.float16(0.1))
    assert np.abs(prob.cpu().numpy() - 1.0 / (1.0 + np.exp(-s))).max() <= 1e-6
