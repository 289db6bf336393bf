"""The trilinear prolongation (Sec. 5.1.1) on its own, against exact rational
arithmetic: a full periodic level, coarse corrections of widely spread size
and sign with zeros and subnormals among them, phi = 0 before the step, so
that the result is the interpolated value itself.

FP64 forms 64 x a child's value as one integer sum at the scale
2^(E - 1078), E the largest biased exponent of the eight coarse values, and
rounds it once: the error of 64 x the value is at most half an ulp of it plus
63 units of that scale (the weights other than the largest operand's); values
all below 2^-960, or above 2^1009, take the nested form, three roundings of
intermediate sums up to 64 x the largest value.  FP32 takes that form
always."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cmg():
    import __graft_entry__ as ge
    ge.build()
    from paper_2604_06035_gb300 import cmg as _c
    return _c


@pytest.fixture(scope="module")
def level(cmg):
    from paper_2604_06035_gb300 import inputs
    ctx = cmg.cmg_ctx_create(0)
    lv = cmg.cmg_level_build(ctx, 3, cmg.cmg_morton_encode(ctx, inputs.uniform_oct_coords(3)))
    yield lv
    cmg.cmg_ctx_destroy(ctx)


def _coarse(kind, rng):
    v = rng.normal(size=(4, 4, 4))
    if kind == "spread":
        v *= np.exp2(rng.integers(-70, 70, size=v.shape))
    elif kind == "zeros":
        v[rng.uniform(size=v.shape) < 0.6] = 0.0
        v[0, 0, 0], v[1, 2, 3] = -0.0, 5e-324
    elif kind == "one_sign":
        v = np.abs(v) + 1.0
    elif kind == "tiny":
        v *= 1e-300
    elif kind == "huge":
        v *= 2.0 ** 1012
    return v


def _exact(coarse, cell):
    """(64 x value, the eight operands) of a fine cell."""
    total, ops = Fraction(0), []
    for t in range(8):
        at, w = [], 1
        for a in range(3):
            f = cell[a] >> 1
            toward = 1 if cell[a] & 1 else -1
            if (t >> a) & 1:
                at.append((f + toward) % 4)
            else:
                at.append(f)
                w *= 3
        x = float(coarse[tuple(at)])
        ops.append(x)
        total += w * Fraction(x)
    return total, ops


@pytest.mark.parametrize("kind", ["plain", "spread", "zeros", "one_sign", "tiny", "huge"])
@pytest.mark.parametrize("colour1_only", [False, True])
def test_fp64_prolongation_matches_exact_interpolation(cmg, level, kind, colour1_only):
    from paper_2604_06035_gb300 import inputs
    coarse = _coarse(kind, np.random.default_rng(11))
    cmg.cmg_level_mg_set(level, 1, 0, inputs.dense_to_octs(coarse, inputs.uniform_oct_coords(2)))
    cmg.cmg_level_mg_set(level, 0, 0, np.zeros((64, 8)))
    if colour1_only:
        cmg.cmg_level_mg_step_range(level, 0, 3, 1, 0, 64)
    else:
        cmg.cmg_level_mg_step(level, 0, 3)
    got = inputs.octs_to_dense(cmg.cmg_level_mg_get(level, 0, 0), inputs.uniform_oct_coords(3), 8)
    for cell in np.ndindex(8, 8, 8):
        if colour1_only and sum(cell) % 2 == 0:
            assert got[cell] == 0.0
            continue
        want, ops = _exact(coarse, cell)
        big = max(abs(x) for x in ops)
        if kind in ("tiny", "huge"):
            bound = 64 * 8 * Fraction(np.spacing(big))  # nested roundings
        else:
            near = float(abs(want))
            bound = Fraction(np.spacing(near)) / 2 + 63 * Fraction(np.spacing(big)) / 8
        assert abs(64 * Fraction(float(got[cell])) - want) <= bound, cell


def test_fp32_prolongation_matches_exact_interpolation(cmg, level):
    from paper_2604_06035_gb300 import inputs
    coarse = _coarse("spread", np.random.default_rng(12))
    coarse = (np.sign(coarse) * np.abs(coarse) ** 0.2).astype(np.float32)
    cmg.cmg_level_solve(level, precision=cmg.CMG_PREC_MIXED, fixed_cycles=1)  # makes the FP32 fields
    oc = inputs.uniform_oct_coords(2)
    cmg.cmg_level_mg_set(level, 1, 0, inputs.dense_to_octs(coarse, oc), precision=cmg.CMG_PREC_MIXED)
    cmg.cmg_level_mg_set(level, 0, 0, np.zeros((64, 8), np.float32), precision=cmg.CMG_PREC_MIXED)
    cmg.cmg_level_mg_step(level, 0, 3, precision=cmg.CMG_PREC_MIXED)
    got = inputs.octs_to_dense(cmg.cmg_level_mg_get(level, 0, 0, cmg.CMG_PREC_MIXED), inputs.uniform_oct_coords(3), 8)
    for cell in np.ndindex(8, 8, 8):
        want, ops = _exact(coarse, cell)
        bound = 64 * 8 * Fraction(float(np.spacing(np.float32(max(abs(x) for x in ops)))))
        assert abs(64 * Fraction(float(got[cell])) - want) <= bound, cell
