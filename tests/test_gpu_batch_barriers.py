"""Which levels of a batched FP64 solve the blocks work on by themselves, seen
from the grid barriers it reports.  The expected count follows from the rule:
patches dealt out to the blocks in contiguous ranges by the middle of each in
the level's octs, and the blocks on their own from the first coarse level on
which none has more octs than threads.  Patches that touch at a corner, whose
prolongation reads the other patch, keep a grid barrier after every operation."""
import numpy as np
import pytest

from test_gpu_batch_own import _box, _patches

pytestmark = pytest.mark.gpu


def _octs_per_level(coords, depth):
    """Octs of a patch on each multigrid level: the parents of the fully
    active octs of the level below."""
    octs = {tuple(c): 0xFF for c in coords.tolist()}
    out = [len(octs)]
    for _ in range(depth - 1):
        up = {}
        for (x, y, z), m in octs.items():
            if m == 0xFF:
                p = (x >> 1, y >> 1, z >> 1)
                up[p] = up.get(p, 0) | 1 << ((x & 1) + 2 * (y & 1) + 4 * (z & 1))
        octs = up
        out.append(len(octs))
    return out


def _split(counts, depth, grid, threads):
    n = len(counts)
    for m in range(1, depth):
        start = np.concatenate([[0], np.cumsum([c[m] for c in counts])])
        block = [min(grid - 1, (int(start[k]) + int(start[k + 1])) // 2 * grid // int(start[n])) for k in range(n)]
        load = np.bincount(block, weights=np.diff(start), minlength=grid)
        if load.max() <= threads:
            return m
    return depth


@pytest.mark.parametrize("kind", ["few", "many", "large", "corner"])
@pytest.mark.parametrize("threads,per_sm,n_pre,n_post", [(256, 2, 2, 2), (32, 1, 1, 2), (512, 1, 2, 0)])
def test_grid_barriers(kind, threads, per_sm, n_pre, n_post):
    import torch

    import __graft_entry__ as ge
    ge.build()
    from paper_2604_06035_gb300 import cmg
    patches = _patches(kind)
    coords = np.concatenate(patches)
    offsets = np.concatenate([[0], np.cumsum([len(p) for p in patches])]).astype(np.int64)
    ctx = cmg.cmg_ctx_create(0)
    P = cmg.cmg_level_build(ctx, 7, cmg.cmg_morton_encode(ctx, _box((0, 0, 0), (64, 64, 64))))
    F = cmg.cmg_level_build(ctx, 8, cmg.cmg_morton_encode(ctx, coords), parent=P)
    cmg.cmg_level_set_density(F, np.random.default_rng(9).uniform(0.2, 1.8, (len(coords), 8)), 1.0)
    B = cmg.cmg_batch_create(F, offsets)
    cmg.cmg_batch_set_schedule(B, threads=threads, blocks_per_sm=per_sm, n_pre=n_pre, n_post=n_post, inner_cycles=1)
    depth = cmg.cmg_level_mg_depth(F)
    counts = [_octs_per_level(p, depth) for p in patches]
    assert [sum(c[m] for c in counts) for m in range(depth)] == [cmg.cmg_level_mg_info(F, m)[0] for m in range(depth)]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    split = depth if kind == "corner" else _split(counts, depth, sms * per_sm, threads)
    assert kind == "corner" or split < depth

    cycles = 2
    _, st = cmg.cmg_batch_solve(B, tol=1e-10, fixed_cycles=cycles)
    down = min(split, depth - 1)
    cycle = down * (2 * n_pre + 1 + 1 + 2 * n_post) + (1 if split < depth else 2 * (n_pre + n_post))
    # set-up, ||f||, scales, ||r||; the test of every cycle and of the end
    assert st["grid_barriers"] == 4 + (cycles + 1) + cycles * (cycle + 1)
    cmg.cmg_ctx_destroy(ctx)
