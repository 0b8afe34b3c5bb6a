"""A bounded wait of the flagger that runs out reaches every kind of caller: the calls that only queue
work return, rfi_status reports it once, and no Adam step is taken while it stands.  The wait is the
self-test's, on a barrier that nothing completes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp32", [False, True])
def test_a_wait_that_ran_out_is_reported_and_stops_training(fp32):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0910_1517_gb300 import build, corr
    build.build()
    corr.load()
    st = torch.cuda.current_stream()
    rng = np.random.default_rng(3)
    x = torch.from_numpy(rng.normal(size=(2, 64, 64)).astype(np.float16)).cuda()
    m = torch.from_numpy((rng.random((2, 64, 64)) < 0.1).astype(np.uint8)).cuda()
    prob = torch.empty((2, 64, 64), device="cuda")
    p0 = (rng.normal(size=9441) * 0.1).astype(np.float32)
    net = (corr.rfi_create_fp32 if fp32 else corr.rfi_create)(2)
    try:
        corr.rfi_set_params(net, p0)
        corr.rfi_infer(net, x, 2, prob, stream=st)
        corr.rfi_status(net, st)
        good = prob.cpu().numpy()
        corr.rfi_wait_selftest(net)
        corr.rfi_train_step(net, x, m, 2, 1e-2, stream=st)         # queued: returns, and changes nothing
        corr.rfi_infer(net, x, 2, prob, stream=st)
        with pytest.raises(corr.CorrError) as ei:
            corr.rfi_status(net, st)
        assert ei.value.code == -8
        corr.rfi_status(net, st)                                   # reported once
        assert np.array_equal(corr.rfi_get_params(net), p0)
        assert np.array_equal(prob.cpu().numpy(), good)
        corr.rfi_train_step(net, x, m, 2, 1e-2, want_loss=True, stream=st)
        assert not np.array_equal(corr.rfi_get_params(net), p0)
    finally:
        corr.rfi_destroy(net)
