"""Where the U-Net's fields lie does not show in its results: outputs that
overlap inputs or each other, at any offset, get what separate arrays get, and
host arrays in a call on device memory (or the reverse) are read like the
rest.  Inference repeats itself bit for bit, so the comparison is exact."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

D, B = 32, 2
N = B * D ** 3


@pytest.fixture(scope="module")
def setup():
    import torch

    import __graft_entry__ as ge
    ge.build()
    from oracle import unet_oracle as U
    from paper_2604_06035_gb300 import cmg
    ctx = cmg.cmg_ctx_create(0)
    net = cmg.cmg_unet_create(ctx, D, B)
    params = U.init_params(3)
    params[-17:-1] = np.random.default_rng(4).normal(0, 0.3, 16)
    cmg.cmg_unet_set_params(net, params.astype(np.float32))
    g = torch.Generator(device="cuda").manual_seed(5)
    rho, field, base, target = (torch.randn((4, N), generator=g, device="cuda")[k].contiguous() for k in range(4))
    yield cmg, net, rho.abs() + 0.5, field, base, target
    cmg.cmg_ctx_destroy(ctx)


def _ptr(t):
    return None if t is None else C.c_void_p(t.data_ptr())


@pytest.mark.parametrize("kernels", [1, 0])
@pytest.mark.parametrize("case", ["pred on base", "delta on base", "pred past base", "delta before base",
                                  "pred on field", "delta on field", "pred on rho", "delta past pred", "both one"])
def test_overlapping_outputs(setup, kernels, case):
    import torch
    cmg, net, rho, field, base, _ = setup
    cmg.cmg_unet_set_kernels(net, kernels)
    want = [torch.empty(N, device="cuda") for _ in range(2)]
    own_base = None if "field" in case else base
    ok = cmg.lib().cmg_unet_forward(net.h, _ptr(rho), _ptr(field), _ptr(own_base), B, _ptr(want[0]), _ptr(want[1]), 1)
    assert ok == cmg.CMG_OK

    # one array with room around the named field; the other output apart
    room, off = 4097, {"on": 0, "past": 4097, "before": -4097, "one": 0}[case.split()[1]]
    big = torch.zeros(N + 2 * room, device="cuda")
    name = case.split()[-1]
    at = big[room:room + N]
    fields = {"rho": rho, "field": field, "base": own_base}
    if name in fields:
        at.copy_(fields[name])
        fields[name] = at
    moved = big[room + off:room + off + N]
    apart = torch.empty(N, device="cuda")
    out = {"pred": (moved, apart), "delta": (apart, moved), "both": (at, at)}[case.split()[0]]
    if name == "pred":
        out = (at, moved)
    rc = cmg.lib().cmg_unet_forward(net.h, _ptr(fields["rho"]), _ptr(fields["field"]), _ptr(fields["base"]), B,
                                    _ptr(out[0]), _ptr(out[1]), 1)
    assert rc == cmg.CMG_OK
    torch.cuda.synchronize()
    cmg.cmg_unet_set_kernels(net, 1)
    assert torch.equal(out[1], want[1])  # written last
    if name == "pred":
        assert torch.equal(out[0][:off], want[0][:off])
    elif case != "both one":
        assert torch.equal(out[0], want[0])


@pytest.mark.parametrize("on_host", ["base", "target", "field base target", "rho", "rho field"])
def test_host_and_device_arrays_in_one_call(setup, on_host):
    import torch
    cmg, net, rho, field, base, target = setup
    shape = (B, D, D, D)
    a = {"rho": rho, "field": field, "base": base, "target": target}
    want = cmg.cmg_unet_forward(net, rho.view(shape), field.view(shape), base=base.view(shape)).cpu()
    loss = cmg.cmg_unet_gradients(net, rho.view(shape), field.view(shape), target.view(shape),
                                  base=base.view(shape))[0].item()
    a = {k: v.view(shape).cpu().numpy() if k in on_host.split() else v.view(shape) for k, v in a.items()}
    if (("rho" in on_host) == ("field" in on_host)):
        got = cmg.cmg_unet_forward(net, a["rho"], a["field"], base=a["base"])
        got = got.cpu() if torch.is_tensor(got) else torch.from_numpy(got)
        assert torch.equal(got, want)
    # the loss of a host call is the mean, that of a device call the sum: FP64
    # sums of 2 D^3 squares in any order, 2^-53 each
    got = cmg.cmg_unet_gradients(net, a["rho"], a["field"], a["target"], base=a["base"])[0]
    got = got.item() if torch.is_tensor(got) else got * N
    assert abs(got - loss) <= N * 2.0 ** -53 * loss
