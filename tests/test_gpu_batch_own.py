"""Batched solves whose coarse levels each block works on by itself: patches so
small that this begins right below the top, several patches per block, blocks
without one, one large patch among small ones, and patches that touch at a
corner (whose prolongation reads the other patch, so that the grid barriers
stay).  With n_pre + n_post coarsest sweeps the batch does what the solve of
the whole level does: two FP64 cycles to 1e-12 of the oracle's, mixed precision
and CG to the same solution."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cmg():
    import __graft_entry__ as ge
    ge.build()
    from paper_2604_06035_gb300 import cmg as _c
    return _c


def _box(lo, size):
    r = [np.arange(a, a + s) for a, s in zip(lo, size)]
    return np.stack(np.meshgrid(*r, indexing="ij"), -1).reshape(-1, 3).astype(np.uint32)


def _patches(kind):
    rng = np.random.default_rng(3)
    at = [(16 * i + 1, 16 * j + 1, 16 * k + 1) for i in range(8) for j in range(8) for k in range(8)]
    if kind == "few":
        return [_box(at[k], s) for k, s in ((0, (1, 1, 1)), (70, (2, 2, 2)), (300, (5, 4, 3)))]
    if kind == "many":
        return [_box(at[k], rng.integers(1, 6, size=3)) for k in range(400)]
    if kind == "large":
        return [_box((3, 3, 3), (25, 27, 26))] + [_box(at[k], rng.integers(2, 6, size=3)) for k in range(300, 330)]
    return [_box((8, 8, 8), (8, 8, 8)), _box((16, 16, 16), (8, 8, 8)), _box((80, 80, 80), (3, 3, 3))]  # corner


@pytest.mark.parametrize("kind", ["few", "many", "large", "corner"])
@pytest.mark.parametrize("threads,per_sm,n_pre,n_post", [(256, 2, 2, 2), (32, 1, 1, 2), (512, 1, 2, 0)])
def test_own_levels_match_the_oracle(cmg, kind, threads, per_sm, n_pre, n_post):
    patches = _patches(kind)
    coords = np.concatenate(patches)
    offsets = np.concatenate([[0], np.cumsum([len(p) for p in patches])]).astype(np.int64)
    rng = np.random.default_rng(9)
    rho = rng.uniform(0.2, 1.8, (len(coords), 8))
    pc = _box((0, 0, 0), (64, 64, 64))
    pphi = rng.normal(size=(len(pc), 8))
    ctx = cmg.cmg_ctx_create(0)
    P = cmg.cmg_level_build(ctx, 7, cmg.cmg_morton_encode(ctx, pc))
    cmg.cmg_level_set_phi(P, pphi)
    F = cmg.cmg_level_build(ctx, 8, cmg.cmg_morton_encode(ctx, coords), parent=P)
    cmg.cmg_level_set_density(F, rho, 1.0)
    B = cmg.cmg_batch_create(F, offsets)
    cmg.cmg_batch_set_schedule(B, threads=threads, blocks_per_sm=per_sm, n_pre=n_pre, n_post=n_post, inner_cycles=1)
    RP = O.Level(7, O.morton_encode(pc))
    RP.set_phi(pphi)
    R = O.Level(8, O.morton_encode(coords), parent=RP)
    R.set_density(rho, 1.0)

    zero = np.zeros_like(rho)
    prm = dict(n_pre=n_pre, n_post=n_post, coarse_sweeps=n_pre + n_post)
    rc, _ = cmg.cmg_batch_solve(B, tol=1e-10, fixed_cycles=2)
    assert rc == cmg.CMG_OK
    R.solve(tol=1e-10, fixed_cycles=2, **prm)
    phi, ref = cmg.cmg_level_get_phi(F), R.get_phi()
    assert np.max(np.abs(phi - ref)) <= 1e-12 * np.max(np.abs(ref))
    R.solve(tol=1e-13, max_cycles=200, **prm)
    ref = R.get_phi()
    for krylov in (0, 1):
        cmg.cmg_level_set_phi(F, zero)
        rc, st = cmg.cmg_batch_solve(B, tol=1e-11, max_cycles=200, precision=cmg.CMG_PREC_MIXED, krylov=krylov)
        assert rc == cmg.CMG_OK and st["n_converged"] == len(patches)
        assert np.max(np.abs(cmg.cmg_level_get_phi(F) - ref)) <= 1e-9 * np.max(np.abs(ref))
    cmg.cmg_ctx_destroy(ctx)
