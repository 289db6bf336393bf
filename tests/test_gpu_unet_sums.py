"""Weight gradients of the U-Net at 64^3 with 8 samples against recorded ones.

The order in which a weight's products are summed shows in its last bits (the
tensor cores truncate as they accumulate) and, through Adam, in every later
step of a training run, so the recorded order is kept.  What differs from run
to run is the order of the FP32 additions that join the sums of up to 607 runs
of bricks: each rounds by 2.5e-8 of the sum so far (the standard deviation of
half a unit in the last place, averaged over a binade), sqrt(607 / 3) times
that over all of them, 3.5e-7, and 5e-7 for the difference of two such sums.
The bound is twice that, over 128 weights of a layer; sums in another order
were 3e-6 to 4e-6 away in the layers on the large grids.

The recorded values come from inputs that are exact in FP32 and made of
integers, so that every machine has the same."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

D, B, SAMPLES, BOUND = 64, 8, 128, 1e-6
LAYERS = [(16, 16), (16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (96, 32), (32, 32), (48, 16), (16, 16)]
RECORD = os.path.join(os.path.dirname(__file__), "golden", "unet_weight_gradients_64x8.txt")


def inputs():
    rng = np.random.default_rng(20)
    v = [rng.integers(0, 256, (B, D, D, D)) for _ in range(3)]
    rho = (0.5 + v[0] / 256.0).astype(np.float32)
    field = ((v[1] - 128) / 64.0).astype(np.float32)
    target = (field + (v[2] - 100) / 128.0 + (v[0] - 128) / 256.0).astype(np.float32)
    parts = []
    for k, (ci, co) in enumerate(LAYERS):
        w = rng.integers(-128, 128, (co, 27, ci)) / 128.0 * np.sqrt(6.0 / (27 * ci))
        if k == 0:
            w[:, :, 2:] = 0.0
        parts += [w.ravel(), rng.integers(0, 256, co) / 512.0]  # positive: no dead layer
    parts += [rng.integers(-128, 128, 16) / 256.0, np.array([0.015625])]
    return rho, field, target, np.concatenate(parts).astype(np.float32)


def gradients(cmg):
    """{layer: 128 of its weights' gradients} of the first pass."""
    rho, field, target, params = inputs()
    ctx = cmg.cmg_ctx_create(0)
    net = cmg.cmg_unet_create(ctx, D, B)
    cmg.cmg_unet_set_params(net, params)
    _, g = cmg.cmg_unet_gradients(net, rho, field, target)
    cmg.cmg_ctx_destroy(ctx)
    out, o = {}, 0
    for k, (ci, co) in enumerate(LAYERS):
        w = g[o:o + co * 27 * ci].reshape(co, 27, ci)[:, :, :2 if k == 0 else ci].ravel()
        out[k] = w[(np.arange(SAMPLES) * 7919 + 5) % len(w)]
        o += co * 27 * ci + co
    return out


def test_weight_gradients_repeat_recorded_ones():
    import __graft_entry__ as ge
    ge.build()
    from paper_2604_06035_gb300 import cmg
    got = gradients(cmg)
    off = {}
    for line in open(RECORD):
        k, words = int(line.split()[0]), line.split()[1:]
        ref = np.array([int(w, 16) for w in words], dtype=np.uint32).view(np.float32).astype(np.float64)
        assert len(ref) == SAMPLES
        assert np.linalg.norm(ref) > 0.0
        off[k] = np.linalg.norm(got[k] - ref) / np.linalg.norm(ref)
    assert len(off) == len(LAYERS) and all(v <= BOUND for v in off.values()), off
