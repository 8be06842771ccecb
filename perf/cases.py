"""The calls a user of this package makes, as cases that can be timed and checked.

A case is one call (or one short sequence of calls) through the package's public entry points:
hard-binned MI of one pose, of a one-parameter sweep, of a registration step's finite differences, of
thousands of poses in one batch and of an uneven batch of pairs; Parzen MI with its gradient for one
pose, for many and over several pairs; a random-sampling metric; the allocation-free call; and a
context that is created for a single evaluation.  Volumes are head-like layered ellipsoids with Rician
noise, the moving one a non-monotonic remap of the same anatomy under a known motion.
"""
from __future__ import annotations

import atexit
import math
import os
import tempfile

import numpy as np
import torch

import paper_1909_10690_gb300 as mi

DEV = "cuda"
MOTION = (6.0, -4.0, 3.0, 4.0, -3.0, 6.0, 1.04, 0.97, 1.02)  # mm, degrees, factors
OVERLAP = 0.82  # typical share of the fixed voxels inside the moving volume, for work()
_KEPT = {}  # the temporary folder of this process's autotune file


def _case(name, call, nx, ny, nz, dtype, depth, bins, n, q, poses, **more):
    c = {"name": name, "call": call, "nx": nx, "ny": ny, "nz": nz, "mx": nx, "my": ny, "mz": nz, "sz": 1.0,
         "dtype": dtype, "depth": depth, "bins": bins, "n": n, "q": q, "poses": poses, "transform": "params",
         "rotation": "euler", "scale": "factor", "form": "additive", "log_bits": False, "fraction": 0.0,
         "on_gpu": False, "entropies": True, "pairs": 1}
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: one pose of the tiny ellipsoid workload's size
        _case("one_pose_64", "eval", 64, 64, 64, "uint8", 8, 32, 1, "1", "near"),
        # one pose of the full-histogram pair
        _case("one_pose_256", "eval", 256, 256, 256, "uint16", 12, 256, 1, "0.5,1,1.5,2", "near"),
        # one parameter swept in 81 steps over the head pair, six q from each histogram
        _case("sweep_head", "eval", 256, 256, 160, "uint16", 12, 128, 81, "0.5,0.8,1,1.2,1.5,2", "sweep", sz=1.2),
        # an iteration of the Kiefer-Wolfowitz registration: 16 poses x 18 central differences on a cropped fixed volume
        _case("registration_step", "eval", 144, 144, 96, "uint16", 12, 64, 288, "1,1.5", "kw", mx=192, my=192, mz=128,
              sz=1.2, entropies=False),
        # thousands of poses of the full-histogram pair in one call
        _case("batch_256", "eval", 256, 256, 256, "uint16", 12, 256, 4096, "0.5,1,1.5,2", "wide", on_gpu=True),
        # pairs of unequal sizes, types and bin counts, 64 poses each
        _case("uneven_pairs", "batch_eval", 96, 96, 96, "mixed", 12, 128, 64, "0.5,1,1.5,2", "wide", pairs=12),
        # the metric over a random quarter of the voxels, unit-ball rotations
        _case("sampled", "eval", 192, 192, 128, "uint16", 12, 64, 400, "1", "wide", rotation="versor", scale="offset",
              fraction=0.25, on_gpu=True),
        # Parzen MI and gradient: one pose, the 50 poses of the differentiable workload, several pairs at once
        _case("gradient_one", "grad", 192, 192, 128, "float32", 0, 64, 1, "1", "near", sz=1.2),
        _case("gradient_50", "grad", 192, 192, 128, "float32", 0, 64, 50, "1,0.7,1.3", "wide", sz=1.2, on_gpu=True),
        _case("gradient_pairs", "batch_grad", 96, 96, 96, "mixed", 12, 128, 8, "1,0.7,1.3", "near", pairs=6),
        # no allocation on the request path
        _case("noalloc", "noalloc", 192, 192, 128, "uint16", 12, 64, 1, "1,1.5", "near", sz=1.2, on_gpu=True),
        # a new pair evaluated once: context, evaluation, release
        _case("new_pair", "new_pair", 192, 160, 128, "uint16", 12, 64, 1, "1", "near", on_gpu=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _types(rng):
    return rng.choice([("uint8", 8), ("uint16", 12), ("uint16", 16), ("float32", 0)])


def draw(rng):
    call = rng.choice(["eval", "eval", "eval", "eval", "batch_eval", "grad", "grad", "batch_grad", "noalloc", "new_pair"])
    dims = [_log_int(rng, 40, 288) for _ in range(3)]
    dtype, depth = _types(rng)
    qs = rng.choice(["1", "1", "1,1.5", "0.5,1,2", "1,0.7,1.3", "0.5,0.8,1,1.2,1.5,2"])
    more = {"sz": rng.choice([1.0, 1.2]), "on_gpu": rng.random() < 0.5, "entropies": rng.random() < 0.5}
    if rng.random() < 0.3:  # a moving volume of another size
        more.update({k: _log_int(rng, 40, 288) for k in ("mx", "my", "mz")})
    voxels = dims[0] * dims[1] * dims[2]
    if call in ("batch_eval", "batch_grad"):
        pairs = rng.randint(2, 8)
        n = _log_int(rng, 1, 96 if call == "batch_eval" else 12)
        return _unnamed(_case("", call, 96, 96, 96, "mixed", 12, 128, n, "1,0.7,1.3" if call == "batch_grad" else qs,
                              "near" if call == "batch_grad" else "wide", pairs=pairs, sz=1.0,
                              on_gpu=more["on_gpu"], entropies=more["entropies"]))
    if call == "grad":
        n = max(1, min(_log_int(rng, 1, 64), int(3e8 / voxels)))
        bins = rng.choice([16, 32, 64, 64, 96, 128])
        more["transform"] = rng.choice(["params", "params", "affine"])
        return _unnamed(_case("", call, *dims, dtype, depth, bins, n, "1,0.7,1.3" if len(qs) > 10 else qs, "near", **more))
    if call == "noalloc":
        dtype, depth = rng.choice([("uint8", 8), ("uint16", 12), ("uint16", 16)])
        more["on_gpu"] = True
        return _unnamed(_case("", call, *dims, dtype, depth, rng.choice([32, 64, 64, 128, 256]), 1, qs, "near", **more))
    bins = rng.choice([32, 64, 64, 128, 256])
    if call == "new_pair":
        return _unnamed(_case("", call, *dims, dtype, depth, bins, 1, qs, "near", **more))
    n = max(1, min(_log_int(rng, 1, 4096), int(1.2e10 / voxels)))
    more.update(rng.choice([{}, {}, {"transform": "affine"}, {"rotation": "versor", "scale": "offset"}]))
    more.update(rng.choice([{}, {}, {"form": "pseudo_additive"}, {"log_bits": True}]))
    if rng.random() < 0.15:
        more["fraction"] = rng.choice([0.1, 0.25, 0.5])
    return _unnamed(_case("", call, *dims, dtype, depth, bins, n, qs, rng.choice(["wide", "near", "sweep"]), **more))


def _unnamed(case):
    case.pop("name")
    return case


def _qs(case):
    return [float(np.float32(v)) for v in case["q"].split(",")]  # the library takes q in 32 bits


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _rotation(rx, ry, rz):
    a, b, c = np.deg2rad([rx, ry, rz])
    x = np.array([[1, 0, 0], [0, np.cos(a), -np.sin(a)], [0, np.sin(a), np.cos(a)]])
    y = np.array([[np.cos(b), 0, np.sin(b)], [0, 1, 0], [-np.sin(b), 0, np.cos(b)]])
    z = np.array([[np.cos(c), -np.sin(c), 0], [np.sin(c), np.cos(c), 0], [0, 0, 1]])
    return z @ y @ x


def _head(rng, extent):
    """Ellipsoids (centre relative to the volume's, quadratic form, class) of a layered head of this extent (mm)."""
    def solid(c, axes, angles):
        r = _rotation(*angles)
        return np.asarray(c), r @ np.diag(1.0 / np.asarray(axes) ** 2) @ r.T

    c, form = solid(rng.uniform(-0.02, 0.02, 3) * extent, extent * np.array([0.36, 0.42, 0.40]), rng.uniform(-6, 6, 3))
    out = [(c, form, 1), (c, form / 0.81, 2), (c, form / 0.74, 3), (c, form / 0.49, 4)]
    for k in range(7):
        far, large = (0.12, 0.08) if k < 3 else (0.2, 0.06)
        out.append((*solid(c + rng.uniform(-far, far, 3) * extent, rng.uniform(0.03, large, 3) * extent,
                           rng.uniform(-90, 90, 3)), 2 if k < 3 else 3))
    return out


def _render(head, means, dims, spacing, motion, dtype, depth, gen):
    """The head's class means with Rician noise on a grid, seen through a motion about the volume centre (or None)."""
    axes = [(torch.arange(d, device=DEV, dtype=torch.float32) - (d - 1) / 2) * s for d, s in zip(dims, spacing)]
    linear, shift = (np.eye(3), np.zeros(3)) if motion is None else (_rotation(*motion[3:6]) @ np.diag(motion[6:9]),
                                                                      np.asarray(motion[:3]))
    inverse = np.linalg.inv(linear)
    volume = torch.full((dims[2], dims[1], dims[0]), float(means[0]), device=DEV)
    x, y, z = axes[0][None, None, :], axes[1][None, :, None], axes[2][:, None, None]
    for c, form, cls in head:
        centre, f = linear @ c + shift, inverse.T @ form @ inverse
        dx, dy, dz = x - float(centre[0]), y - float(centre[1]), z - float(centre[2])
        r = (float(f[0, 0]) * dx * dx + 2 * float(f[0, 1]) * dx * dy + float(f[1, 1]) * dy * dy) \
            + (2 * float(f[0, 2]) * dx + 2 * float(f[1, 2]) * dy + float(f[2, 2]) * dz) * dz
        volume[r <= 1.0] = float(means[cls])
    noise = 0.02
    volume.add_(torch.randn(volume.shape, device=DEV, generator=gen), alpha=noise)
    volume = torch.hypot(volume, torch.randn(volume.shape, device=DEV, generator=gen) * noise)
    if dtype == "float32":
        return volume.clamp_(0.0, 1.0)
    full = float((1 << depth) - 1)
    return (volume * full).round_().clamp_(0.0, full).to(torch.int32).to(torch.uint8 if dtype == "uint8" else torch.uint16)


def _specs(case, seed):
    """Geometry, type and bins of each pair of the case."""
    if case["dtype"] != "mixed":
        return [dict(dims=(case["nx"], case["ny"], case["nz"]), mdims=(case["mx"], case["my"], case["mz"]),
                     spacing=(1.0, 1.0, case["sz"]), dtype=case["dtype"], depth=case["depth"], bins=case["bins"])]
    rng = np.random.default_rng(7)  # sizes belong to the case, not to the inputs
    out = []
    for i in range(case["pairs"]):
        dims = (96, 96, 96) if i == 0 else (320, 320, 200) if i == 1 else tuple(
            int(rng.integers(96, hi + 1)) for hi in (320, 320, 200))
        u8 = i % 2 == 0
        out.append(dict(dims=dims, mdims=dims, spacing=(1.0, 1.0, 1.0), dtype="uint8" if u8 else "uint16",
                        depth=8 if u8 else 12, bins=int(rng.choice([32, 64, 128]))))
    return out


def _volumes(case, seed):
    out = []
    for i, s in enumerate(_specs(case, seed)):
        rng = np.random.default_rng([seed, i])
        gen = torch.Generator(device=DEV).manual_seed(1000 * (seed % 1000003) + i)
        extent = np.array([min(d, m) for d, m in zip(s["dims"], s["mdims"])]) * np.asarray(s["spacing"])
        if case["poses"] == "kw":  # the fixed volume is a centred crop: the head has the moving volume's extent
            extent = np.array(s["mdims"]) * np.asarray(s["spacing"])
        head = _head(rng, extent)
        t1 = [0.0, rng.uniform(0.08, 0.15), rng.uniform(0.15, 0.25), rng.uniform(0.45, 0.55), rng.uniform(0.7, 0.8)]
        t2 = [0.0, rng.uniform(0.05, 0.10), rng.uniform(0.8, 0.9), rng.uniform(0.5, 0.6), rng.uniform(0.3, 0.38)]
        fixed = _render(head, t1, s["dims"], s["spacing"], None, s["dtype"], s["depth"], gen)
        moving = _render(head, t2, s["mdims"], s["spacing"], MOTION, s["dtype"], s["depth"], gen)
        out.append((s, fixed, moving))
    return out


def _poses(case, seed):
    """n x 9 (or n x 12) float32 parameters."""
    rng = np.random.default_rng([seed, 77])
    n = case["n"] * (case["pairs"] if case["dtype"] == "mixed" else 1)
    p = np.empty((n, 9), np.float64)
    if case["poses"] == "wide":
        p[:, :3], p[:, 3:6] = rng.uniform(-15, 15, (n, 3)), rng.uniform(-20, 20, (n, 3))
        p[:, 6:] = rng.uniform(0.85, 1.15, (n, 3))
    elif case["poses"] == "sweep":
        p[:] = (0, 0, 0, 0, 0, 0, 1, 1, 1)
        axis = int(rng.integers(9))
        lo, hi = ((-20, 20), (-30, 30), (0.8, 1.2))[axis // 3]
        p[:, axis] = np.linspace(lo, hi, n) + rng.uniform(-0.01, 0.01)
    else:  # near the known motion
        starts = max(1, n // 18) if case["poses"] == "kw" else n
        p0 = np.asarray(MOTION) + np.concatenate([rng.uniform(-4, 4, (starts, 3)), rng.uniform(-5, 5, (starts, 3)),
                                                  rng.uniform(-0.04, 0.04, (starts, 3))], axis=1)
        if case["poses"] == "kw":  # +- c along every parameter of every pose
            step = np.diag([0.5] * 6 + [0.005] * 3)
            p0 = (p0[:, None, :] + np.concatenate([step, -step])[None]).reshape(-1, 9)
        p[:] = p0[np.arange(n) % len(p0)]
    if case["transform"] == "affine":
        out = np.empty((n, 3, 4))
        for t in range(n):
            out[t, :, :3], out[t, :, 3] = _rotation(*p[t, 3:6]) @ np.diag(p[t, 6:]), p[t, :3]
        return out.reshape(n, 12).astype(np.float32)
    if case["rotation"] == "versor":
        p[:, 3:6] = np.sin(np.deg2rad(p[:, 3:6]) / 2)
    if case["scale"] == "offset":
        p[:, 6:] -= 1.0
    return p.astype(np.float32)


# ---------------------------------------------------------------------------
# The calls
# ---------------------------------------------------------------------------

def _context_args(case):
    return dict(kernel="parzen" if "grad" in case["call"] else "hard", tsallis_form=case["form"],
                bits=case["log_bits"], rotation=case["rotation"], scale=case["scale"], transform=case["transform"],
                sample_fraction=case["fraction"], sample_seed=11)


def _pair_args(s, fixed, moving):
    return dict(fixed=fixed, moving=moving, bins=s["bins"], fixed_spacing=s["spacing"], moving_spacing=s["spacing"],
                fixed_depth=s["depth"] or None, moving_depth=s["depth"] or None)


def _keep_tuning():
    """The batched path's autotuned choices are kept in a file, as a program that makes many contexts keeps them."""
    if "dir" not in _KEPT:
        _KEPT["dir"] = tempfile.TemporaryDirectory(prefix="mi_tuned_")
        atexit.register(_KEPT["dir"].cleanup)
        mi.autotune_cache(os.path.join(_KEPT["dir"].name, "tuned"))


def prepare(case, seed):
    _keep_tuning()
    volumes = _volumes(case, seed)
    poses = _poses(case, seed)
    state = {"call": case["call"], "q": _qs(case), "entropies": case["entropies"], "args": _context_args(case)}
    if case["call"] in ("noalloc", "new_pair"):
        state["pair"] = _pair_args(*volumes[0])
        state["poses"] = poses
        return state
    if case["dtype"] == "mixed":
        pair_of = np.repeat(np.arange(case["pairs"], dtype=np.int32), case["n"])
        state["pair_of"] = torch.from_numpy(pair_of).to(DEV) if case["on_gpu"] else pair_of
        state["ctx"] = mi.Context(pairs=[_pair_args(*v) for v in volumes], **state["args"])
    else:
        state["ctx"] = mi.Context(**_pair_args(*volumes[0]), **state["args"])
    put = (lambda a: torch.from_numpy(a).to(DEV)) if case["on_gpu"] else (lambda a: a)
    # the context has served a call of this size on other poses before
    state["poses"] = put(_poses(case, seed + 1))
    run(state)
    state["poses"] = put(poses)
    return state


def run(state):
    call, q, poses = state["call"], state["q"], state["poses"]
    if call == "eval":
        out = state["ctx"].eval(poses, q, with_entropies=state["entropies"])
    elif call == "batch_eval":
        out = state["ctx"].batch_eval(state["pair_of"], poses, q, with_entropies=state["entropies"])
    elif call == "grad":
        out = state["ctx"].grad(poses, q, allow_empty=True)
    elif call == "batch_grad":
        out = state["ctx"].batch_grad(state["pair_of"], poses, q, allow_empty=True)
    elif call == "noalloc":
        out = mi.eval_noalloc(transform=poses[0], q=q, **state["pair"])
    else:
        ctx = mi.Context(**state["pair"], **state["args"])
        out = ctx.eval(poses, q, with_entropies=state["entropies"])
        ctx.close()
    return out


def work(case):
    """Each volume read once, parameters in, results out; 20 integer operations a voxel of the overlap (three
    coordinates, seven lerps, two bins, weights, address, increment), or for the Parzen form 31 FP32 operations
    forward and 32 + 19 per q in the adjoint."""
    size = {"uint8": 1, "uint16": 2, "float32": 4}
    nq, pairs = len(_qs(case)), _specs(case, 0)
    voxels = sum(s["dims"][0] * s["dims"][1] * s["dims"][2] for s in pairs)
    nbytes = sum((s["dims"][0] * s["dims"][1] * s["dims"][2] + s["mdims"][0] * s["mdims"][1] * s["mdims"][2])
                 * size[s["dtype"]] for s in pairs)
    n = case["n"] * len(pairs)
    grad = "grad" in case["call"]
    nparams = 12 if case["transform"] == "affine" else 9
    nbytes += n * (4 * nparams + 8 * nq * ((1 + nparams) if grad else 4 if case["entropies"] else 1))
    per_voxel = 31 + 32 + 19 * nq if grad else 20
    share = case["fraction"] if case["fraction"] > 0 else 1.0
    return {"bytes": float(nbytes), "flops": float(per_voxel * OVERLAP * share * voxels * case["n"])}


# ---------------------------------------------------------------------------
# The same results in 64 bits
# ---------------------------------------------------------------------------

def _turn(axis, angle, derivative=False):
    c, s = math.cos(angle), math.sin(angle)
    m = np.zeros((3, 3))
    a, b = (axis + 1) % 3, (axis + 2) % 3
    if derivative:
        m[a, a], m[a, b], m[b, a], m[b, b] = -s, -c, c, -s
    else:
        m[axis, axis], m[a, a], m[a, b], m[b, a], m[b, b] = 1.0, c, -s, s, c
    return m


def _linear(case, p):
    """The 3 x 3 motion matrix and translation of one pose, with their derivatives by parameter (Euler or affine)."""
    if case["transform"] == "affine":
        m = p.reshape(3, 4)
        dm, dt = np.zeros((12, 3, 3)), np.zeros((12, 3))
        for a in range(3):
            for c in range(3):
                dm[4 * a + c, a, c] = 1.0
            dt[4 * a + 3, a] = 1.0
        return m[:, :3], m[:, 3], dm, dt
    sigma = p[6:9] + (1.0 if case["scale"] == "offset" else 0.0)
    dm, dt = np.zeros((9, 3, 3)), np.zeros((9, 3))
    if case["rotation"] == "versor":
        x, y, z = p[3:6]
        n2 = x * x + y * y + z * z
        if n2 >= 1.0:
            x, y, z = p[3:6] / math.sqrt(n2)
        w = math.sqrt(1.0 - n2) if n2 < 1.0 else 0.0
        r = np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                      [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                      [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])
    else:
        unit = math.pi / 180.0
        angle = p[3:6] * unit
        r = _turn(2, angle[2]) @ _turn(1, angle[1]) @ _turn(0, angle[0])
        for k in range(3):
            t = [_turn(a, angle[a], a == k) for a in range(3)]
            dm[3 + k] = (t[2] @ t[1] @ t[0]) * unit * sigma
    for k in range(3):
        dt[k, k] = 1.0
        dm[6 + k][:, k] = r[:, k]
    return r * sigma, p[:3], dm, dt


def _index_affine(case, s, p):
    """[A | b] from fixed to moving index, and its derivatives (P x 3 x 4)."""
    m, t, dm, dt = _linear(case, p.astype(np.float64))
    sp = np.asarray(np.float32(s["spacing"]), np.float64)
    cf, cm = sp * (np.asarray(s["dims"]) - 1) * 0.5, sp * (np.asarray(s["mdims"]) - 1) * 0.5
    out = np.empty((3, 4))
    out[:, :3], out[:, 3] = m * sp / sp[:, None], (cm + t - m @ cf) / sp
    d = np.empty((len(dm), 3, 4))
    d[:, :, :3], d[:, :, 3] = dm * sp / sp[:, None], (dt - dm @ cf) / sp
    return out, d


def _fixed_point(a, bits):
    s = np.abs(a) * float(1 << bits)
    return (np.sign(a) * np.floor(s + 0.5)).astype(np.int64)


def _positions(A, dims, mdims, bits, keep):
    """Fixed-point moving indices of the fixed voxels inside the moving volume, and those voxels' linear indices."""
    i, j, k = (torch.arange(d, device=DEV, dtype=torch.int64) for d in dims)
    U, inside = [], keep
    for a in range(3):
        u = (int(A[a, 0]) * i)[None, None, :] + (int(A[a, 1]) * j)[None, :, None] + (int(A[a, 2]) * k + int(A[a, 3]))[:, None, None]
        ok = (u >= 0) & (u <= (mdims[a] - 1) << bits)
        inside = ok if inside is None else inside & ok
        U.append(u)
    at = inside.reshape(-1).nonzero().squeeze(1)
    return [u.reshape(-1)[at] for u in U], at


def _integers(v, s):
    if s["dtype"] == "float32":
        return (v.double() * 65535.0).round().clamp(0, 65535).to(torch.int64), 16
    return v.to(torch.int32).to(torch.int64), s["depth"]


def _sampled(case, s):
    if not case["fraction"]:
        return None

    def mix(x):
        x = x ^ (x >> 16)
        x = (x * 0x85EBCA6B) & 0xFFFFFFFF
        x = x ^ (x >> 13)
        x = (x * 0xC2B2AE35) & 0xFFFFFFFF
        return x ^ (x >> 16)

    n = s["dims"][0] * s["dims"][1] * s["dims"][2]
    seed = int(mix(torch.tensor(11, dtype=torch.int64)))
    limit = int(math.floor(float(np.float32(case["fraction"])) * 4294967296.0))
    keep = mix(torch.arange(n, device=DEV, dtype=torch.int64) ^ seed) < limit
    return keep.reshape(s["dims"][2], s["dims"][1], s["dims"][0])


def _entropy(p, q, log_bits):
    p = p[p > 0]
    if q == 1.0:
        h = -(p * p.log()).sum()
        return h / math.log(2.0) if log_bits else h
    return (1.0 - (p ** q).sum()) / (q - 1.0)


def _mi(P, q, case):
    f, m, j = (_entropy(x, q, case["log_bits"]) for x in (P.sum(1), P.sum(0), P.reshape(-1)))
    v = f + m - j
    if q != 1.0 and case["form"] == "pseudo_additive":
        v = v + (1.0 - q) * f * m
    return v, torch.stack([f, m, j])


def _exact_hard(case, s, fixed, moving, poses):
    fv, fdepth = _integers(fixed, s)
    mv, mdepth = _integers(moving, s)
    fb, mv = ((fv * s["bins"]) >> fdepth).reshape(-1), mv.reshape(-1)
    nx, ny, nz = s["mdims"]
    keep, B = _sampled(case, s), s["bins"]
    mi_out, h_out, counts = [], [], []
    for p in poses:
        A = _fixed_point(_index_affine(case, s, p)[0], 16)
        U, at = _positions(A, s["dims"], s["mdims"], 16, keep)
        c = [u >> 16 for u in U]
        w = [(u & 0xFFFF) >> 8 for u in U]
        up = [torch.clamp(c[a] + 1, max=s["mdims"][a] - 1) for a in range(3)]

        def lerp(a, b, f):
            return (a * (256 - f) + b * f + 128) >> 8

        planes = []
        for z in (c[2], up[2]):
            rows = [lerp(mv[c[0] + nx * (y + ny * z)], mv[up[0] + nx * (y + ny * z)], w[0]) for y in (c[1], up[1])]
            planes.append(lerp(*rows, w[1]))
        v = lerp(*planes, w[2])
        H = torch.bincount(fb[at] * B + ((v * B) >> mdepth), minlength=B * B).reshape(B, B).double()
        N = H.sum()
        counts.append(int(N))
        got = [_mi(H / N, q, case) for q in _qs(case)]
        mi_out.append(torch.stack([g[0] for g in got]))
        h_out.append(torch.stack([g[1] for g in got]))
    return torch.stack(mi_out), torch.stack(h_out), torch.tensor(counts)


def _unit(v, s):
    return v.double().clamp(0, 1) if s["dtype"] == "float32" else v.to(torch.int32).double() / ((1 << s["depth"]) - 1)


def _exact_parzen(case, s, fixed, moving, poses):
    B, (nx, ny, nz) = s["bins"], s["mdims"]
    if s["dtype"] == "float32":
        fb = (fixed.double().clamp(0, 1) * (B - 4)).floor().to(torch.int64) + 2
    else:
        fb = torch.div(fixed.to(torch.int32).to(torch.int64) * (B - 4), (1 << s["depth"]) - 1, rounding_mode="floor") + 2
    fb, mv = fb.reshape(-1), _unit(moving, s).reshape(-1)
    mi_out, g_out = [], []
    for p in poses:
        aff, daff = _index_affine(case, s, p)
        U, at = _positions(_fixed_point(aff, 32), s["dims"], s["mdims"], 32, None)
        N = at.numel()
        c = [torch.clamp(u >> 32, max=m - 2) for u, m in zip(U, s["mdims"])]
        wx, wy, wz = ((u - (k << 32)).double() / 4294967296.0 for u, k in zip(U, c))
        base = c[0] + nx * (c[1] + ny * c[2])
        v = [[[mv[base + x + nx * (y + ny * z)] for x in (0, 1)] for y in (0, 1)] for z in (0, 1)]
        ex = [[v[z][y][1] - v[z][y][0] for y in (0, 1)] for z in (0, 1)]
        ax = [[v[z][y][0] + wx * ex[z][y] for y in (0, 1)] for z in (0, 1)]
        ay = [ax[z][0] + wy * (ax[z][1] - ax[z][0]) for z in (0, 1)]
        m = ay[0] + wz * (ay[1] - ay[0])
        gz = ay[1] - ay[0]
        gy = (1 - wz) * (ax[0][1] - ax[0][0]) + wz * (ax[1][1] - ax[1][0])
        gx = (1 - wz) * (ex[0][0] + wy * (ex[0][1] - ex[0][0])) + wz * (ex[1][0] + wy * (ex[1][1] - ex[1][0]))
        mt = m.clamp(0, 1) * (B - 4) + 2
        k0 = mt.floor().to(torch.int64)
        t = mt - k0
        u = 1 - t
        beta = [u ** 3 / 6, 2 / 3 - t * t + t ** 3 / 2, 2 / 3 - u * u + u ** 3 / 2, t ** 3 / 6]
        slope = [u * u / 2, 2 * t - 1.5 * t * t, 1.5 * u * u - 2 * u, -t * t / 2]
        f = fb[at]
        P = torch.zeros(B * (B + 1), device=DEV, dtype=torch.float64)
        for o in range(4):
            P += torch.bincount(f * (B + 1) + k0 - 1 + o, weights=beta[o], minlength=B * (B + 1))
        P = P.reshape(B, B + 1)[:, :B] / N
        i = at % s["dims"][0]
        j = (at // s["dims"][0]) % s["dims"][1]
        k = at // (s["dims"][0] * s["dims"][1])
        row_mi, row_g = [], []
        for q in _qs(case):
            value, (hf, hm, _) = _mi(P, q, case)
            pf, pm = P.sum(1, keepdim=True).expand(B, B), P.sum(0, keepdim=True).expand(B, B)
            on = P > 0
            if q == 1.0:
                W = (P / (pf * pm)).log() - 1.0
                W = W / math.log(2.0) if case["log_bits"] else W
            else:
                ds = lambda x: -q * x ** (q - 1.0) / (q - 1.0)  # noqa: E731
                W = ds(pf) + ds(pm) - ds(P)
                if case["form"] == "pseudo_additive":
                    W = W + (1.0 - q) * (ds(pf) * hm + hf * ds(pm))
            W = torch.where(on, W, torch.zeros_like(W))
            W = torch.cat([W, torch.zeros(B, 1, device=DEV, dtype=torch.float64)], dim=1).reshape(-1)
            sv = sum(W[f * (B + 1) + k0 - 1 + o] * slope[o] for o in range(4))
            moments = np.empty((3, 4))
            for a, g in enumerate((gx, gy, gz)):
                sg = sv * g
                moments[a] = [float((sg * x).sum()) for x in (i, j, k)] + [float(sg.sum())]
            row_mi.append(value)
            row_g.append(torch.from_numpy(-(B - 4) / N * (daff * moments).sum(axis=(1, 2))))
        mi_out.append(torch.stack(row_mi))
        g_out.append(torch.stack(row_g))
    return torch.stack(mi_out), torch.stack(g_out)


def exact(case, seed):
    grad = "grad" in case["call"]
    volumes, poses, nq = _volumes(case, seed), _poses(case, seed), len(_qs(case))
    cost = sum(s["dims"][0] * s["dims"][1] * s["dims"][2] for s, _, _ in volumes) * case["n"] * (6 + 4 * nq if grad else 1)
    if cost > 9e9:  # over about 20 seconds
        return None
    parts = [(_exact_parzen if grad else _exact_hard)(case, *v, poses[i * case["n"]:(i + 1) * case["n"]])
             for i, v in enumerate(volumes)]
    out = tuple(torch.cat(x) for x in zip(*parts))
    if grad:
        return out
    if case["call"] == "noalloc":
        return out[0][0]
    return out if case["entropies"] else out[0]
