"""FP32 field arrays that start on a 4-byte but not a 16-byte boundary are read
and written like aligned ones, bit for bit."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level", [1, 2, 5])
@pytest.mark.parametrize("shift", [1, 2, 3])
@pytest.mark.parametrize("field", [0, 1])
def test_offset_fp32_arrays(level, shift, field):
    import torch

    import __graft_entry__ as ge
    ge.build()
    from paper_2604_06035_gb300 import cmg, inputs
    coords = inputs.uniform_oct_coords(level)
    n = len(coords)
    values = torch.from_numpy(np.random.default_rng(4).normal(size=8 * n).astype(np.float32)).cuda()
    ctx = cmg.cmg_ctx_create(0)
    lv = cmg.cmg_level_build(ctx, level, cmg.cmg_morton_encode(ctx, coords))
    got = []
    for k in (0, shift):
        src = torch.empty(8 * n + k, device="cuda")[k:]
        src.copy_(values)
        assert src.data_ptr() % 16 == 4 * k
        cmg.cmg_level_mg_set(lv, 0, field, src, precision=cmg.CMG_PREC_MIXED)
        room = torch.full((8 * n + k + 1,), -7.0, device="cuda")
        rc = cmg.lib().cmg_level_mg_get(lv.h, 0, field, cmg.CMG_PREC_MIXED, C.c_void_p(room[k:].data_ptr()),
                                        cmg.CMG_MEM_DEVICE)
        assert rc == cmg.CMG_OK
        cmg.cmg_ctx_synchronize(ctx)
        assert float(room[-1]) == -7.0 and (k == 0 or float(room[k - 1]) == -7.0)
        got.append(room[k:-1].cpu())
    assert torch.equal(got[0], got[1])
    if field == 0:
        assert torch.equal(got[0], values.cpu())
    cmg.cmg_ctx_destroy(ctx)
