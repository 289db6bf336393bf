"""Levels built in memory that other levels left behind: whatever was built,
solved, destroyed or failed to build before on the context, a level's tables,
hierarchy and solutions are bit for bit those of a fresh context.  And the
memory that a context keeps for its levels goes back to the GPU with the last
of them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cmg():
    import __graft_entry__ as ge
    ge.build()
    from paper_2604_06035_gb300 import cmg as _c
    return _c


def _keys(cmg, ctx, coords, bits):
    if bits == 128:
        return cmg.cmg_morton_encode128(ctx, coords.astype(np.uint64))
    return cmg.cmg_morton_encode(ctx, coords)


def _build(cmg, ctx, level, coords, parent, bits):
    build = cmg.cmg_level_build128 if bits == 128 else cmg.cmg_level_build
    return build(ctx, level, _keys(cmg, ctx, coords, bits), parent=parent)


def _ragged(coords, seed):
    """Some of the octs, so that coarse levels are only partly active."""
    keep = np.random.default_rng(seed).random(len(coords)) < 0.8
    return coords[keep]


def _everything(cmg, ctx, base, coords, rho, bits):
    """All that a build makes and a solve in each precision leaves."""
    lv = _build(cmg, ctx, 6, coords, base, bits)
    out = [cmg.cmg_level_get_neighbors(lv), cmg.cmg_level_get_father_cells(lv)]
    for m in range(cmg.cmg_level_mg_depth(lv)):
        keys = cmg.cmg_level_mg_keys128 if bits == 128 else cmg.cmg_level_mg_keys
        out += [keys(lv, m), cmg.cmg_level_mg_active(lv, m)]
    for kw in ({"precision": cmg.CMG_PREC_FP64}, {"precision": cmg.CMG_PREC_MIXED}, {"krylov": 1}):
        cmg.cmg_level_set_density(lv, rho, 1.0)
        cmg.cmg_level_set_phi(lv, np.zeros_like(rho))
        cmg.cmg_level_solve(lv, tol=1e-10, max_cycles=200, **kw)
        out.append(cmg.cmg_level_get_phi(lv))
    cmg.cmg_level_destroy(lv)
    return out


@pytest.mark.parametrize("bits", [64, 128])
def test_rebuilt_levels_repeat_a_fresh_context(cmg, bits):
    from paper_2604_06035_gb300 import inputs
    cfg = inputs.two_level_amr(base_level=5, seed=2)
    bc, fc = cfg["coords"]
    grids = [fc, _ragged(fc, 1), fc[: len(fc) // 3], _ragged(fc, 2)]
    rhos = [np.random.default_rng(k).uniform(0.5, 1.5, (len(c), 8)) for k, c in enumerate(grids)]

    def context():
        ctx = cmg.cmg_ctx_create(0)
        base = _build(cmg, ctx, 5, bc, None, bits)
        cmg.cmg_level_set_density(base, cfg["rho"][0], 1.0)
        cmg.cmg_level_solve(base, tol=1e-10)
        return ctx, base

    fresh = []
    for c, r in zip(grids, rhos):
        ctx, base = context()
        fresh.append(_everything(cmg, ctx, base, c, r, bits))
        cmg.cmg_ctx_destroy(ctx)

    ctx, base = context()
    for round_ in range(2):
        for k in (0, 1, 2, 3, 1, 0):
            # between them, builds that fail: a duplicate key, a key outside
            # the level, and an allocation in the middle
            with pytest.raises(cmg.CmgError):
                _build(cmg, ctx, 6, np.concatenate([grids[k], grids[k][:1]]), base, bits)
            with pytest.raises(cmg.CmgError):
                _build(cmg, ctx, 6, np.concatenate([grids[k], [[32, 0, 0]]]).astype(np.uint32), base, bits)
            cmg.cmg_debug_inject_alloc_failure(7 + 5 * k + round_)
            with pytest.raises(cmg.CmgError):
                _build(cmg, ctx, 6, grids[k], base, bits)
            cmg.cmg_debug_inject_alloc_failure(0)
            got = _everything(cmg, ctx, base, grids[k], rhos[k], bits)
            assert len(got) == len(fresh[k])
            assert all(np.array_equal(a, b) for a, b in zip(got, fresh[k])), (round_, k)
    cmg.cmg_ctx_destroy(ctx)


def test_last_level_gives_the_memory_back(cmg):
    import torch
    from paper_2604_06035_gb300 import inputs
    ctx = cmg.cmg_ctx_create(0)
    coords = inputs.uniform_oct_coords(8)  # 2 M octs: several hundred MiB
    keys = cmg.cmg_morton_encode(ctx, coords)
    small = cmg.cmg_level_build(ctx, 3, cmg.cmg_morton_encode(ctx, inputs.uniform_oct_coords(3)))
    cmg.cmg_level_destroy(small)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for other in (False, True):
        keep = cmg.cmg_level_build(ctx, 3, cmg.cmg_morton_encode(ctx, inputs.uniform_oct_coords(3))) if other else None
        lv = cmg.cmg_level_build(ctx, 8, keys)
        assert torch.cuda.mem_get_info()[0] < free - (256 << 20)
        cmg.cmg_level_destroy(lv)
        if other:  # kept for the next one, within the bound
            assert torch.cuda.mem_get_info()[0] >= free - (640 << 20)
            cmg.cmg_level_destroy(keep)
        assert torch.cuda.mem_get_info()[0] >= free - (64 << 20)
    cmg.cmg_ctx_destroy(ctx)
