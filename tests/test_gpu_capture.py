"""A prediction on device arrays, whose fields are read and written in place, in
a CUDA graph: captured once, replayed on other values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cmg():
    import __graft_entry__ as ge
    ge.build()
    from paper_2604_06035_gb300 import cmg as _c
    return _c


@pytest.mark.parametrize("base_too", [True, False])
def test_prediction_in_a_graph(cmg, base_too):
    import torch
    from oracle import unet_oracle as U
    D, B = 32, 2
    stream = torch.cuda.Stream()
    ctx = cmg.cmg_ctx_create(0, stream)
    net = cmg.cmg_unet_create(ctx, D, B)
    params = U.init_params(3)
    params[-17:-1] = np.random.default_rng(4).normal(0, 0.3, 16)
    cmg.cmg_unet_set_params(net, params.astype(np.float32))
    g = torch.Generator(device="cuda").manual_seed(6)
    rho, field, base, pred, delta = (torch.randn((B, D, D, D), generator=g, device="cuda") for _ in range(5))
    rho = rho.abs() + 0.5
    torch.cuda.synchronize()

    def call():
        rc = cmg.lib().cmg_unet_forward(net.h, rho.data_ptr(), field.data_ptr(), base.data_ptr() if base_too else None,
                                        B, pred.data_ptr(), delta.data_ptr(), cmg.CMG_MEM_DEVICE)
        assert rc == cmg.CMG_OK

    call()  # the weights are prepared once
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        call()
    rho.mul_(1.5)
    field.add_(0.25)
    torch.cuda.synchronize()
    call()
    torch.cuda.synchronize()
    want = pred.clone(), delta.clone()
    pred.zero_()
    delta.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(pred, want[0]) and torch.equal(delta, want[1])
    del graph
    cmg.cmg_ctx_destroy(ctx)
