"""CG on levels around the size from which q = L0 p runs one thread per oct
instead of four (40000 octs), against the oracle's: phi after two iterations
and the residual norms.  The dot products are summed in another order than the
oracle's, which moves alpha and beta at the 1e-16 level: 1e-11 after two
iterations."""
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


# refined octs: 35, 34^3 = 39304 (below), 35^3 = 42875 (above)
@pytest.mark.parametrize("size", [(5, 7, 1), (34, 34, 34), (35, 35, 35)])
def test_two_iterations_match_the_oracle(cmg, size):
    from paper_2604_06035_gb300 import inputs
    rng = np.random.default_rng(6)
    bc = inputs.uniform_oct_coords(6)
    r = [np.arange(2, 2 + s) for s in size]
    fc = np.stack(np.meshgrid(*r, indexing="ij"), -1).reshape(-1, 3).astype(np.uint32)
    rho_b, rho_f = rng.uniform(0.5, 1.5, (len(bc), 8)), rng.uniform(0.5, 1.5, (len(fc), 8))
    rb = float(rho_b.mean())
    ctx = cmg.cmg_ctx_create(0)
    B = cmg.cmg_level_build(ctx, 6, cmg.cmg_morton_encode(ctx, bc))
    F = cmg.cmg_level_build(ctx, 7, cmg.cmg_morton_encode(ctx, fc), parent=B)
    ob = O.Level(6, O.morton_encode(bc))
    of = O.Level(7, O.morton_encode(fc), parent=ob)
    for lv, ol, rho in ((B, ob, rho_b), (F, of, rho_f)):
        cmg.cmg_level_set_density(lv, rho, rb)
        ol.set_density(rho, rb)
        _, st = cmg.cmg_level_solve(lv, fixed_cycles=2, krylov=1)
        _, so = ol.solve_pcg(fixed_cycles=2)
        phi, ref = cmg.cmg_level_get_phi(lv), ol.get_phi()
        assert np.max(np.abs(phi - ref)) <= 1e-11 * np.max(np.abs(ref))
        assert np.allclose(st["rel_history"], so["rel_history"][:2], rtol=1e-9, atol=1e-15)
    cmg.cmg_ctx_destroy(ctx)
