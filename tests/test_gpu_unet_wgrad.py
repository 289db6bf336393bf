"""The weight gradient's kernel against its definition, exactly: with operands
that are small integers every product and every sum (below 2^24) is exact in
FP32, in any order.  Runs of many bricks (the copy ring wraps), of one, and of
unequal length; grids of one brick per axis, whose halo is the brick itself, of
three, and of 48 and 64; every pair of channel counts of the network; the
upsampled and skip inputs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# cin, cout, skip channels
LAYERS = [(16, 16, 0), (16, 32, 0), (32, 32, 0), (32, 64, 0), (64, 64, 0), (96, 32, 32), (48, 16, 16)]
GRIDS = [(4, 1), (4, 700), (8, 3), (12, 5), (16, 8), (32, 9), (48, 2)]


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as ge
    ge.build()
    from paper_2604_06035_gb300 import cmg
    c = cmg.cmg_ctx_create(0)
    yield c
    cmg.cmg_ctx_destroy(c)


def _check(ctx, cin, cout, cb, D, B):
    import torch

    from paper_2604_06035_gb300 import cmg
    g = torch.Generator(device="cuda").manual_seed(1000 * D + B)

    def ints(d, c):
        return torch.randint(-2, 3, (B, d, d, d, c), generator=g, device="cuda").to(torch.bfloat16)

    assert 4 * B * D ** 3 < 2 ** 24
    dout = ints(D, cout)
    skip = ints(D, cb) if cb else None
    inp = ints(D // 2 if cb else D, cin - cb)
    dw, db = cmg.cmg_debug_conv_wgrad(ctx, dout, inp, skip)
    x = inp
    if cb:
        for axis in (1, 2, 3):
            x = x.repeat_interleave(2, dim=axis)
        x = torch.cat([x, skip], dim=-1)
    flat = dout.reshape(-1, cout).float()
    x = x.float()
    old = torch.backends.cuda.matmul.allow_tf32
    torch.backends.cuda.matmul.allow_tf32 = False
    try:
        for t in range(27):
            d = (t // 9 - 1, (t // 3) % 3 - 1, t % 3 - 1)
            shifted = torch.roll(x, tuple(-a for a in d), (1, 2, 3)).reshape(-1, cin)
            assert torch.equal(dw[:, t], flat.T @ shifted), t
    finally:
        torch.backends.cuda.matmul.allow_tf32 = old
    assert torch.equal(db, flat.sum(0))


@pytest.mark.parametrize("D,B", GRIDS)
@pytest.mark.parametrize("cin,cout,cb", LAYERS)
def test_integer_gradients_are_exact(ctx, cin, cout, cb, D, B):
    _check(ctx, cin, cout, cb, D, B)


@pytest.mark.parametrize("cin,cout,cb", [(16, 16, 0), (48, 16, 16), (96, 32, 32)])
def test_integer_gradients_are_exact_at_64(ctx, cin, cout, cb):
    _check(ctx, cin, cout, cb, 64, 8 if cout == 16 else 4)


def test_unsupported_shapes_are_refused(ctx):
    import torch

    from paper_2604_06035_gb300 import cmg
    z = lambda d, c: torch.zeros((1, d, d, d, c), dtype=torch.bfloat16, device="cuda")
    for dout, inp, skip in ((z(8, 48), z(8, 16), None), (z(8, 16), z(8, 24), None), (z(6, 16), z(6, 16), None),
                            (z(8, 16), z(4, 16), z(8, 8))):
        with pytest.raises(cmg.CmgError):
            cmg.cmg_debug_conv_wgrad(ctx, dout, inp, skip)
    with pytest.raises(ValueError):
        cmg.cmg_debug_conv_wgrad(ctx, z(8, 16), z(8, 16), z(8, 16))
