"""What the performance of this library is measured on: the calls a user's program makes, over the
sizes it makes them at.  Every case goes through the public binding (paper_2604_06035_gb300.cmg).

Five kinds of work:

* "chain": a simulation step's gravity.  The AMR levels are built; the step brings new densities,
  solves the periodic base and then every refined level from phi = 0 to a relative residual of
  1e-10 (each level's solve queued behind its parent's), and reads phi back on the device.
  `solver`: FP64 V-cycles, FP32 V-cycles in FP64 refinement ("mixed"), CG preconditioned by a
  V-cycle ("pcg"), or the FFT base with mixed refined levels ("fft").
* "regrid": what an AMR code does after its grid changed: encode the new octs' coordinates, build
  the refined level on its parent (hash, neighbours, ghosts, hierarchy), solve it once, read phi.
* "batch": many independent refined patches solved in one launch, sizes log-uniform.
* "infer" / "train": the learned warm start's network, predicting for a batch of blocks, or one
  training step (loss, gradients, Adam update).

Inputs are made on the GPU from the seed: lognormal densities on k^-2 Gaussian fields, cells above
8 times the mean refined (with one cell of face dilation, properly nested), mass-conserving child
densities; patches are compact irregular balls of octs.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2604_06035_gb300 import cmg

TOL = 1e-10
THRESHOLD = 8.0     # cells denser than this many means are refined
PATCH_LEVEL = 11    # level of the batched patches (each in a 128-oct cube of its own)

# Octs of a refined level per cell of its parent, as the generator below gives them on average
# (work() has the case alone and cannot look at the drawn refinement).
REFINED = {1: 0.09, 2: 0.08, 3: 0.15}


def listed():
    return [
        # the smallest solve: one periodic block, where launches and latency are all there is
        {"name": "base32_fp64", "kind": "chain", "base": 5, "refine": 0, "sigma": 1.0, "solver": "fp64"},
        # the two-level run of an ordinary step, in both precisions users choose between
        {"name": "two128_fp64", "kind": "chain", "base": 7, "refine": 1, "sigma": 1.5, "solver": "fp64"},
        {"name": "two128_mixed", "kind": "chain", "base": 7, "refine": 1, "sigma": 1.5, "solver": "mixed"},
        # the large run: 256^3 base and three refined levels, about 50 million cells
        {"name": "amr256_fp64", "kind": "chain", "base": 8, "refine": 3, "sigma": 2.0, "solver": "fp64"},
        {"name": "amr256_mixed", "kind": "chain", "base": 8, "refine": 3, "sigma": 2.0, "solver": "mixed"},
        # uniform-grid runs take the FFT for their one level
        {"name": "base256_fft", "kind": "chain", "base": 8, "refine": 0, "sigma": 1.5, "solver": "fft"},
        # small AMR run with the Krylov iteration, for operators the plain V-cycle converges slowly on
        {"name": "two64_pcg", "kind": "chain", "base": 6, "refine": 1, "sigma": 1.5, "solver": "pcg"},
        # zoom-in targets solved together: some dozens of middling patches, and the full batch
        {"name": "batch96_mixed", "kind": "batch", "patches": 96, "n_max": 30000, "solver": "mixed"},
        {"name": "batch512_fp64", "kind": "batch", "patches": 512, "n_max": 200000, "solver": "fp64"},
        # the learned warm start on 64^3 blocks: prediction, and a training step
        {"name": "infer64_b8", "kind": "infer", "dim": 64, "blocks": 8},
        {"name": "train64_b8", "kind": "train", "dim": 64, "blocks": 8},
        # the grid changed: rebuild the refined level and solve it
        {"name": "regrid128_mixed", "kind": "regrid", "base": 7, "refine": 1, "sigma": 1.5, "solver": "mixed",
         "key_bits": 64},
    ]


def draw(rng):
    kind = rng.choice(["chain", "chain", "chain", "chain", "batch", "batch", "infer", "train", "train", "regrid"])
    if kind == "chain":
        solver = rng.choice(["fp64", "fp64", "mixed", "mixed", "fft", "pcg"])
        base = rng.randint(4, 8)
        return {"kind": kind, "base": base, "refine": rng.randint(0, 3), "sigma": round(rng.uniform(1.2, 2.0), 3),
                "solver": solver}
    if kind == "regrid":
        return {"kind": kind, "base": rng.randint(5, 8), "refine": 1, "sigma": round(rng.uniform(1.4, 2.0), 3),
                "solver": rng.choice(["fp64", "mixed"]), "key_bits": rng.choice([64, 64, 128])}
    if kind == "batch":
        patches = int(round(math.exp(rng.uniform(math.log(2), math.log(512)))))
        n_max = int(round(math.exp(rng.uniform(math.log(300), math.log(200000)))))
        return {"kind": kind, "patches": patches, "n_max": n_max,
                "solver": rng.choice(["fp64", "mixed", "pcg", "mixed_pcg"])}
    dim = rng.choice([16, 32, 48, 64])
    return {"kind": kind, "dim": dim, "blocks": rng.randint(1, 8)}


# ----------------------------------------------------------------- inputs

def _gen(*seed):
    return torch.Generator(device="cuda").manual_seed(int(np.random.SeedSequence(seed).generate_state(1)[0]))


def _grf(n, g):
    """Periodic unit-rms Gaussian field on n^3 cells [z, y, x], P(k) ~ k^-2 up to the Nyquist mode."""
    w = torch.fft.rfftn(torch.randn((n, n, n), generator=g, dtype=torch.float64, device="cuda"))
    k1 = torch.fft.fftfreq(n, dtype=torch.float64, device="cuda") * n
    kz = torch.fft.rfftfreq(n, dtype=torch.float64, device="cuda") * n
    k = torch.sqrt(k1[:, None, None] ** 2 + k1[None, :, None] ** 2 + kz[None, None, :] ** 2)
    amp = torch.where((k > 0) & (k <= n / 2), 1.0 / k.clamp(min=0.5), torch.zeros_like(k))
    f = torch.fft.irfftn(w * amp, s=(n, n, n))
    f -= f.mean()
    return f / f.square().mean().sqrt()


def _lognormal(n, sigma, g):
    e = torch.exp(sigma * _grf(n, g))
    return e / e.mean()


def _to_octs(dense):
    """[z, y, x] cells -> [n_octs, 8], octs x fastest, child bx + 2 by + 4 bz."""
    m = dense.shape[0] // 2
    return dense.reshape(m, 2, m, 2, m, 2).permute(0, 2, 4, 1, 3, 5).reshape(-1, 8).contiguous()


def _to_dense(octs, m):
    return octs.reshape(m, m, m, 2, 2, 2).permute(0, 3, 1, 4, 2, 5).reshape(2 * m, 2 * m, 2 * m)


def _off():
    c = torch.arange(8, device="cuda")
    return torch.stack([c & 1, (c >> 1) & 1, (c >> 2) & 1], 1)


def _uniform_coords(level):
    r = torch.arange(1 << (level - 1), device="cuda")
    z, y, x = torch.meshgrid(r, r, r, indexing="ij")
    return torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1)


def _lin(c, size):
    return (c[..., 0] * size + c[..., 1]) * size + c[..., 2]


def _refine(level, coords, rho, threshold):
    """Coordinates of the cells to refine, and their places in the level's flattened cells."""
    half, size = 1 << (level - 1), 1 << level
    occ = torch.full((half ** 3,), -1, dtype=torch.int32, device="cuda")
    occ[_lin(coords, half)] = torch.arange(len(coords), dtype=torch.int32, device="cuda")
    flag = rho > threshold
    cells = 2 * coords[:, None, :] + _off()[None]
    dense, marked = cells[flag], flag.clone()
    for axis in range(3):
        for step in (-1, 1):
            q = dense.clone()
            q[:, axis] = (q[:, axis] + step) % size
            o = occ[_lin(q >> 1, half)].long()
            child = (q[:, 0] & 1) + 2 * (q[:, 1] & 1) + 4 * (q[:, 2] & 1)
            marked[o[o >= 0], child[o >= 0]] = True
    cand = marked.reshape(-1).nonzero()[:, 0]
    cc = cells.reshape(-1, 3)[cand]
    ok = torch.ones(len(cand), dtype=torch.bool, device="cuda")
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dz in (-1, 0, 1):
                q = (cc + torch.tensor([dx, dy, dz], device="cuda")) % size
                ok &= occ[_lin(q >> 1, half)] >= 0
    return cc[ok].contiguous(), cand[ok]


def _children(rho_cells, g):
    e = torch.exp(0.5 * torch.randn((len(rho_cells), 8), generator=g, dtype=torch.float64, device="cuda"))
    return rho_cells[:, None] * e / e.mean(1, keepdim=True)


def _chain_inputs(case, seed):
    """[(level, oct coordinates [n, 3], rho [n, 8])] from the base down.  The structure that was refined belongs to the
    case (an AMR code keeps its grid for several steps), placed anywhere in the periodic box by the seed; the densities
    have evolved away from it, each seed's in its own way."""
    grid = _gen(case["base"], int(1000 * case["sigma"]), 1)
    g = _gen(seed, 1)
    shift = torch.tensor(np.random.default_rng([seed, 1]).integers(0, 1 << case["base"], size=3), device="cuda")
    level, n = case["base"], 1 << case["base"]
    field = _grf(n, grid)
    e = torch.exp(case["sigma"] * field)
    coords, rho = _uniform_coords(level), _to_octs(e / e.mean())
    e = torch.exp(case["sigma"] * (0.95 * field + math.sqrt(1 - 0.95 ** 2) * _grf(n, g)))
    e = torch.roll(e / e.mean(), shift.flip(0).tolist(), (0, 1, 2))
    out = [(level, coords, _to_octs(e))]
    for k in range(case["refine"]):
        coords, idx = _refine(level, coords, rho, THRESHOLD)
        if len(coords) == 0:
            break
        rho, level = _children(rho.reshape(-1)[idx], grid), level + 1
        evolved = torch.exp(0.3 * torch.randn(rho.shape, generator=g, dtype=torch.float64, device="cuda"))
        out.append((level, (coords + (shift << k)) % (n << k), rho * evolved))
    return out


def _patch_inputs(case, seed):
    """Patches of log-uniform sizes in [64, n_max] octs at PATCH_LEVEL (the case's; the seed places them), and the
    parent level's octs and phi."""
    sizes = np.random.default_rng([case["patches"], case["n_max"]]).uniform(math.log(64), math.log(case["n_max"]),
                                                                            case["patches"])
    sizes = np.rint(np.exp(sizes)).astype(int)
    rng = np.random.default_rng([seed, 7])
    places = rng.permutation(512)
    g = _gen(seed, 7)
    r = torch.arange(64, device="cuda")
    sub = torch.stack(torch.meshgrid(r, r, r, indexing="ij"), -1).reshape(-1, 3)
    d2 = (sub.double() - 31.5).square().sum(1)
    shapes = [torch.argsort(d2 + 40.0 * torch.rand(len(d2), generator=g, dtype=torch.float64, device="cuda"))
              for _ in range(8)]
    fields = [_lognormal(64, 1.5, g).reshape(-1) for _ in range(8)]
    coords, rho, offsets = [], [], [0]
    for k, n in enumerate(sizes):
        at = shapes[k % 8][:n]
        at_cube = int(places[k])
        cube = torch.tensor([at_cube % 8, (at_cube // 8) % 8, at_cube // 64], device="cuda") * 128 + 32
        coords.append(sub[at] + cube)
        rho.append(fields[(k // 8) % 8][(at + 4099 * k) % 64 ** 3])
        offsets.append(offsets[-1] + int(n))
    coords = torch.cat(coords)
    rho = _children(torch.cat(rho), g)
    half = 1 << (PATCH_LEVEL - 2)
    near = torch.unique(_lin(coords >> 1, half))
    steps = torch.tensor([(a * half + b) * half + c for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)],
                         device="cuda")
    par = torch.unique((near[:, None] + steps[None]).reshape(-1))
    parent = torch.stack([par // (half * half), (par // half) % half, par % half], 1)
    x = (2 * parent[:, None, :] + _off()[None] + 0.5) / (2.0 * half)
    phi = torch.zeros(x.shape[:2], dtype=torch.float64, device="cuda")
    for _ in range(8):
        kv = torch.tensor(rng.integers(-2, 3, size=3), dtype=torch.float64, device="cuda")
        phi += rng.normal() * torch.sin(2 * math.pi * (x.double() @ kv) + rng.uniform(0, 6.28))
    return coords, np.array(offsets, dtype=np.int64), rho, parent, phi


def _unet_inputs(case, seed):
    """rho, field, base, target [B, D, D, D]: the target adds to the base a smooth linear map of the field, as the
    change of a potential is one of its residual."""
    D, B = case["dim"], case["blocks"]
    g = _gen(seed, D, B, 3)
    rho, field, base, target = [], [], [], []
    k = torch.fft.fftfreq(D, dtype=torch.float64, device="cuda") * D
    sym = sum(torch.sin(math.pi * a / D).square() for a in (k[:, None, None], k[None, :, None], k[None, None, :]))
    sym[0, 0, 0] = 1.0
    for _ in range(B):
        r = _lognormal(D, 1.5, g)
        f = r * _grf(D, g)
        f = f - f.mean()
        e = torch.fft.ifftn(torch.fft.fftn(f) / sym).real
        b = _grf(D, g)
        rho.append(r)
        field.append(f)
        base.append(b)
        target.append(b + f.square().mean().sqrt() * (e - e.mean()) / e.std())
    return [torch.stack(v).float().contiguous() for v in (rho, field, base, target)]


LAYERS = [(16, 16), (16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (96, 32), (32, 32), (48, 16), (16, 16)]


def _unet_params(seed):
    """He-normal weights, small biases; the padding channels of the first layer unused."""
    rng = np.random.default_rng([seed, 11])
    parts = []
    for k, (ci, co) in enumerate(LAYERS):
        w = rng.normal(0.0, math.sqrt(2.0 / (27 * ci)), size=(co, 27, ci))
        if k == 0:
            w[:, :, 2:] = 0.0
        parts += [w.ravel(), rng.normal(0.0, 0.05, size=co)]
    parts += [rng.normal(0.0, 0.2, size=16), rng.normal(0.0, 0.05, size=1)]
    return np.concatenate(parts).astype(np.float32)


# ------------------------------------------------- what a program has in hand

def _build(ctx, level, coords, parent=None, key_bits=64):
    if key_bits == 128:
        return cmg.cmg_level_build128(ctx, level, cmg.cmg_morton_encode128(ctx, coords), parent=parent)
    return cmg.cmg_level_build(ctx, level, cmg.cmg_morton_encode(ctx, coords), parent=parent)


def _coords_arg(coords, key_bits=64):
    if key_bits == 128:
        return coords.contiguous().view(torch.uint64)
    return coords.to(torch.int32).contiguous().view(torch.uint32)


def _params(solver, base):
    kind = {"fp64": cmg.CMG_PREC_FP64, "pcg": cmg.CMG_PREC_FP64, "mixed": cmg.CMG_PREC_MIXED,
            "mixed_pcg": cmg.CMG_PREC_MIXED, "fft": cmg.CMG_PREC_FFT if base else cmg.CMG_PREC_MIXED}[solver]
    return cmg.solve_params(tol=TOL, max_cycles=200, precision=kind, krylov=int(solver.endswith("pcg")))


def prepare(case, seed):
    ctx = cmg.cmg_ctx_create(0)
    if case["kind"] in ("chain", "regrid"):
        levels, parent = [], None
        inputs = _chain_inputs(case, seed)
        bits = case.get("key_bits", 64)
        for k, (level, coords, rho) in enumerate(inputs):
            if case["kind"] == "regrid" and k == 1:
                break
            parent = _build(ctx, level, _coords_arg(coords, bits), parent, bits)
            levels.append((parent, rho, torch.zeros_like(rho), _params(case["solver"], k == 0)))
        if case["kind"] == "chain":
            return {"kind": "chain", "ctx": ctx, "levels": levels}
        lv, rho, zero, _ = levels[0]
        cmg.cmg_level_set_density(lv, rho, 1.0)
        cmg.cmg_level_solve(lv, _params("mixed", True))
        # a base without a cell over the threshold refines its middle eighth
        if len(inputs) > 1:
            level, coords, rho = inputs[1]
        else:
            m = 1 << (case["base"] - 1)
            level, rho = case["base"] + 1, torch.ones((m ** 3, 8), dtype=torch.float64, device="cuda")
            coords = _uniform_coords(case["base"]) + m // 2
        return {"kind": "regrid", "ctx": ctx, "parent": lv, "level": level, "bits": bits,
                "coords": _coords_arg(coords, bits), "rho": rho, "params": _params(case["solver"], False)}
    if case["kind"] == "batch":
        coords, offsets, rho, pcoords, pphi = _patch_inputs(case, seed)
        parent = _build(ctx, PATCH_LEVEL - 1, _coords_arg(pcoords))
        cmg.cmg_level_set_phi(parent, pphi)
        lv = _build(ctx, PATCH_LEVEL, _coords_arg(coords), parent)
        batch = cmg.cmg_batch_create(lv, offsets)
        cmg.cmg_batch_set_schedule(batch, threads=256, blocks_per_sm=2, n_pre=2, n_post=3, inner_cycles=1)
        return {"kind": "batch", "ctx": ctx, "level": lv, "batch": batch, "rho": rho, "zero": torch.zeros_like(rho),
                "params": _params(case["solver"], False)}
    rho, field, base, target = _unet_inputs(case, seed)
    net = cmg.cmg_unet_create(ctx, case["dim"], case["blocks"])
    cmg.cmg_unet_set_params(net, _unet_params(seed))
    return {"kind": case["kind"], "ctx": ctx, "net": net, "rho": rho, "field": field, "base": base, "target": target}


def run(state):
    kind = state["kind"]
    if kind == "chain":
        for lv, rho, zero, params in state["levels"]:
            cmg.cmg_level_set_density(lv, rho, 1.0)
            cmg.cmg_level_set_phi(lv, zero)
            cmg.cmg_level_solve_async(lv, params)
        for lv, _, _, _ in state["levels"]:
            cmg.cmg_level_solve_wait(lv)
        return [cmg.cmg_level_get_phi(lv, device=True) for lv, _, _, _ in state["levels"]]
    if kind == "regrid":
        lv = _build(state["ctx"], state["level"], state["coords"], state["parent"], state["bits"])
        cmg.cmg_level_set_density(lv, state["rho"], 1.0)
        cmg.cmg_level_solve(lv, state["params"])
        out = [cmg.cmg_level_get_neighbors(lv, device=True), cmg.cmg_level_get_father_cells(lv, device=True),
               cmg.cmg_level_get_phi(lv, device=True)]
        cmg.cmg_level_destroy(lv)
        return out
    if kind == "batch":
        cmg.cmg_level_set_density(state["level"], state["rho"], 1.0)
        cmg.cmg_level_set_phi(state["level"], state["zero"])
        cmg.cmg_batch_solve(state["batch"], state["params"])
        return cmg.cmg_level_get_phi(state["level"], device=True)
    if kind == "infer":
        return cmg.cmg_unet_forward(state["net"], state["rho"], state["field"], base=state["base"])
    loss, grads = cmg.cmg_unet_gradients(state["net"], state["rho"], state["field"], state["target"],
                                         base=state["base"])
    cmg.cmg_unet_adam_step(state["net"], 1e-4)
    return [loss, grads, cmg.cmg_unet_get_params(state["net"], device=True)]


def work(case):
    """Minimum traffic: densities and the initial phi read, phi written (8 bytes a cell each); for the network its
    inputs and outputs and 27-tap convolutions.  Flops of the solves: the sweeps, residual and grid transfers of the
    V-cycles that 1e-10 takes at a factor of ten a cycle."""
    if case["kind"] in ("infer", "train"):
        D, B = case["dim"], case["blocks"]
        vox = [D ** 3, D ** 3 // 8, D ** 3 // 64]
        flops = B * sum(54.0 * ci * co * vox[lvl] for (ci, co), lvl in zip(LAYERS, (0, 0, 1, 1, 2, 2, 1, 1, 0, 0)))
        n = sum(27 * ci * co + co for ci, co in LAYERS) + 17
        if case["kind"] == "infer":
            return {"bytes": 16.0 * B * vox[0] + 4.0 * n, "flops": flops}
        return {"bytes": 16.0 * B * vox[0] + 4.0 * n * 8, "flops": 3.0 * flops}
    if case["kind"] == "batch":
        octs = case["patches"] * (case["n_max"] - 64) / math.log(case["n_max"] / 64.0)
    else:
        octs, level_octs = 0.0, 8.0 ** (case["base"] - 1)
        for k in range(case["refine"] + 1):
            octs += level_octs if case["kind"] == "chain" or k else 0.0
            level_octs *= 8 * REFINED.get(k + 1, 0.1)
    cells = 8.0 * octs
    if case.get("solver") == "fft" and case["refine"] == 0:
        return {"bytes": 24.0 * cells, "flops": cells * (2 * 2 * 2.5 * 3 * case["base"] + 3 * 10)}
    extra = 4.0 * 3 * octs + 4.0 * 19 * octs if case["kind"] == "regrid" else 0.0
    return {"bytes": 24.0 * cells + extra, "flops": cells * 10 * (4 * 7 + 9 + 5) * 8 / 7}


# ------------------------------------------------------------------- 64 bits

def _poisson_periodic(rho_octs, level):
    n = 1 << level
    f = _to_dense(rho_octs - 1.0, n // 2)
    s = torch.sin(math.pi * torch.fft.fftfreq(n, dtype=torch.float64, device="cuda")).square()
    sr = torch.sin(math.pi * torch.fft.rfftfreq(n, dtype=torch.float64, device="cuda")).square()
    sym = -4.0 * n * n * (s[:, None, None] + s[None, :, None] + sr[None, None, :])
    sym[0, 0, 0] = 1.0
    fh = torch.fft.rfftn(f) / sym
    fh[0, 0, 0] = 0.0
    return _to_octs(torch.fft.irfftn(fh, s=(n, n, n)))


class _Cells:
    """Lookup of a level's cells by coordinates."""

    def __init__(self, coords, level):
        self.size, self.n = 1 << level, 8 * len(coords)
        self.cells = (2 * coords[:, None, :] + _off()[None]).reshape(-1, 3)
        self.keys, self.order = torch.sort(_lin(self.cells, self.size))

    def find(self, q):
        k = _lin(q % self.size, self.size)
        at = torch.searchsorted(self.keys, k).clamp(max=self.n - 1)
        return torch.where(self.keys[at] == k, self.order[at], self.n)


def _poisson_refined(coords, level, rho, parent, parent_phi):
    """The refined level's discrete solution by conjugate gradients in 64 bits, its boundary interpolated from the
    parent's phi."""
    C = _Cells(coords, level)
    b = -(rho.reshape(-1) - 1.0) / float(C.size) ** 2
    nbs = []
    pphi = torch.cat([parent_phi.reshape(-1), torch.zeros(1, dtype=torch.float64, device="cuda")])
    for axis in range(3):
        for step in (-1, 1):
            q = C.cells.clone()
            q[:, axis] += step
            nb = C.find(q)
            gone = (nb == C.n).nonzero()[:, 0]
            gq = q[gone] % C.size
            side = 2 * (gq & 1) - 1
            val = torch.zeros(len(gone), dtype=torch.float64, device="cuda")
            for t in range(8):
                bits = torch.tensor([t & 1, (t >> 1) & 1, (t >> 2) & 1], device="cuda")
                w = 0.75 ** (3 - int(bits.sum())) * 0.25 ** int(bits.sum())
                val += w * pphi[parent.find((gq >> 1) + side * bits)]
            b[gone] += val
            nbs.append(nb.to(torch.int32))
    x = torch.zeros_like(b)
    r, p = b.clone(), torch.zeros(C.n + 1, dtype=torch.float64, device="cuda")
    p[:-1] = r
    rr = torch.dot(r, r)
    stop = 1e-28 * float(rr)
    for it in range(3000):
        q = 6.0 * p[:-1]
        for nb in nbs:
            q -= p[nb]
        a = rr / torch.dot(p[:-1], q)
        x += a * p[:-1]
        r -= a * q
        new = torch.dot(r, r)
        if it % 16 == 15 and float(new) <= stop:
            break
        p[:-1] = r + (new / rr) * p[:-1]
        rr = new
    return x.reshape(-1, 8), C


def _unet_exact(case, seed):
    rho, field, base, target = [v.double() for v in _unet_inputs(case, seed)]
    flat = torch.from_numpy(_unet_params(seed)).double().cuda().requires_grad_(case["kind"] == "train")
    at = [0]

    def take(*shape):
        n = int(np.prod(shape))
        at[0] += n
        return flat[at[0] - n:at[0]].reshape(shape)

    def conv(x):
        ci, co = LAYERS[len(done)]
        w = take(co, 3, 3, 3, ci).permute(0, 4, 1, 2, 3)
        done.append(1)
        return F.relu(F.conv3d(F.pad(x, (1,) * 6, mode="circular"), w, take(co)))

    done = []
    dims = (1, 2, 3)
    rms = field.square().mean(dims, keepdim=True).sqrt()
    x = torch.zeros((len(rho), 16) + tuple(rho.shape[1:]), dtype=torch.float64, device="cuda")
    x[:, 0] = (rho - rho.mean(dims, keepdim=True)) / rho.std(dims, keepdim=True, unbiased=False)
    x[:, 1] = field / rms
    s0 = conv(conv(x))
    s1 = conv(conv(F.avg_pool3d(s0, 2)))
    u = conv(conv(F.avg_pool3d(s1, 2)))
    u = conv(conv(torch.cat([F.interpolate(u, scale_factor=2), s1], 1)))
    u = conv(conv(torch.cat([F.interpolate(u, scale_factor=2), s0], 1)))
    hw, hb = take(16), take(1)
    delta = (u * hw[None, :, None, None, None]).sum(1) + hb
    if case["kind"] == "infer":
        return base + rms * delta
    sq = (delta - (target - base) / rms).square()
    sq.mean().backward()
    g = flat.grad
    new = flat.detach() - 1e-4 * g / (g.abs() + 1e-8)  # Adam's first step, bias-corrected
    return [sq.sum().detach().reshape(1), g, new]


def exact(case, seed):
    if case["kind"] in ("infer", "train"):
        return _unet_exact(case, seed)
    if case["kind"] == "batch":
        if case["patches"] * case["n_max"] > 20000000:  # too many cells for the plain iteration in the time
            return None
        coords, _, rho, pcoords, pphi = _patch_inputs(case, seed)
        return _poisson_refined(coords, PATCH_LEVEL, rho, _Cells(pcoords, PATCH_LEVEL - 1), pphi)[0]
    out, cells = [], None
    for k, (level, coords, rho) in enumerate(_chain_inputs(case, seed)):
        if k == 0:
            out.append(_poisson_periodic(rho, level))
            cells = _Cells(coords, level)
        else:
            phi, cells = _poisson_refined(coords, level, rho, cells, out[-1])
            out.append(phi)
    if case["kind"] == "regrid":
        return [None, None, out[1]] if len(out) > 1 else None
    return out
