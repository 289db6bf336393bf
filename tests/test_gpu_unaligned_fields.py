"""Field arrays that start on an 8-byte (FP32: 4-byte) but not a 16-byte
boundary are read and written like aligned ones, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level", [1, 2, 5])
def test_offset_device_arrays(level):
    import torch

    import __graft_entry__ as ge
    ge.build()
    from paper_2604_06035_gb300 import cmg, inputs
    coords = inputs.uniform_oct_coords(level)
    n = len(coords)
    rng = np.random.default_rng(3)
    rho, phi = rng.uniform(0.5, 1.5, (n, 8)), rng.normal(size=(n, 8))
    ctx = cmg.cmg_ctx_create(0)

    def offset(a, dtype):
        t = torch.empty(8 * n + 1, dtype=dtype, device="cuda")[1:]
        if a is not None:
            t.copy_(torch.from_numpy(np.ascontiguousarray(a)).reshape(-1))
        return t.view(n, 8)

    got = []
    for at in (lambda a: torch.from_numpy(a).cuda(), lambda a: offset(a, torch.float64)):
        lv = cmg.cmg_level_build(ctx, level, cmg.cmg_morton_encode(ctx, coords))
        cmg.cmg_level_set_density(lv, at(rho), float(rho.mean()))
        cmg.cmg_level_set_phi(lv, at(phi))
        out = offset(None, torch.float64)
        cmg.cmg_level_get_phi(lv, out=out)
        f = cmg.cmg_level_mg_get(lv, 0, 1)
        cmg.cmg_ctx_synchronize(ctx)
        got.append((out.cpu().numpy(), f))
    assert np.array_equal(got[0][0], phi) and np.array_equal(got[1][0], phi)
    assert np.array_equal(got[0][1], got[1][1])
    cmg.cmg_ctx_destroy(ctx)
