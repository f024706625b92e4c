"""What this framework is timed on: the work its users have it do, through the public entry points.

Every case is one planner-side call (or the few calls that belong together) on data already on the
GPU: candidate scans on a 2D map in the three variants, trajectories, the map update, depth-camera
batches in a voxel map, run-length encoding, a mixed stream of candidate sets, and the learned
surrogate's inference and training step. The sizes are those of the repository's benchmark and tests
(random 200x200 grid, 2048x2048 office map, 512x512x128 voxel map, 4096 candidates, batches of 4096
beams) and generic odd ones around them; draw() spreads further cases over the same ranges.

exact() recomputes each result in 64 bits with plain torch from the paper's formulas.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1905_02238_gb300 import fsmi, surrogate, synth

VARIANTS = {"exact": fsmi.EXACT, "approx": fsmi.APPROX, "uniform": fsmi.UNIFORM}
DOCC, DEMP = 1.5, 0.67


def listed():
    return [
        # one scan of a small robot's local map: the smallest call, all latency and launches
        {"name": "scan_200", "kind": "eval2d", "W": 200, "H": 200, "world": "random", "P": 1, "B": 360, "R": 64.0,
         "variant": "exact", "sigma": 1.5, "band": 3, "e0": 0},
        # a planner scoring candidate poses on an explored building, exact FSMI: the benchmark's batch
        {"name": "office_exact", "kind": "eval2d", "W": 2048, "H": 2048, "world": "office", "P": 1024, "B": 360,
         "R": 256.0, "variant": "exact", "sigma": 2.0, "band": 6, "e0": 0},
        # Approx-FSMI with the paper's Delta = 3 on a cropped map, odd counts, the no-return event kept
        {"name": "office_approx_odd", "kind": "eval2d", "W": 1531, "H": 1187, "world": "office", "P": 517, "B": 181,
         "R": 181.5, "variant": "approx", "sigma": 1.5, "band": 3, "e0": 1},
        # the same planner with uniform noise, the cheapest variant: traversal and gathers dominate
        {"name": "office_uniform", "kind": "eval2d", "W": 2048, "H": 2048, "world": "office", "P": 1024, "B": 360,
         "R": 256.0, "variant": "uniform", "sigma": 2.0, "band": 4, "e0": 0},
        # discretised candidate trajectories with cells counted once per trajectory (Section 2.4)
        {"name": "trajectories", "kind": "traj", "W": 1024, "H": 1024, "world": "office", "T": 48, "S": 16, "B": 180,
         "R": 128.0, "sigma": 2.0},
        # the Bayesian update of the map by a short buffer of scans
        {"name": "map_update", "kind": "update", "W": 1024, "H": 1024, "world": "office", "P": 32, "B": 720,
         "R": 200.0},
        # depth-camera views in a voxel map, FSMI-RLE: the benchmark's 3D batch
        {"name": "voxels_exact", "kind": "eval3d", "X": 512, "Y": 512, "Z": 128, "P": 64, "rw": 128, "rh": 128,
         "R": 384, "variant": "exact", "reading": 0, "sigma": 2.0, "band": 6, "cap": 64},
        # Theorem 5 on a smaller volume of odd extents with a coarse camera
        {"name": "voxels_thm5_odd", "kind": "eval3d", "X": 301, "Y": 253, "Z": 77, "P": 23, "rw": 80, "rh": 61,
         "R": 200, "variant": "approx", "reading": 0, "sigma": 2.0, "band": 6, "cap": 64},
        # the two-step 3D path: rays encoded once, then evaluated (and kept for further evaluations)
        {"name": "encode_then_eval", "kind": "encode", "X": 256, "Y": 256, "Z": 96, "P": 12, "rw": 96, "rh": 96,
         "R": 256, "variant": "uniform", "reading": 0, "sigma": 2.0, "band": 4, "cap": 64},
        # a stream of candidate sets of both kinds and many ranges in one call
        {"name": "mixed_sets", "kind": "mixed", "W": 1024, "H": 1024, "X": 192, "Y": 192, "Z": 64, "sets": 64,
         "pmax2": 96, "pmax3": 6, "B": 360, "rw": 64, "rh": 64, "rmax2": 128, "rmax3": 128, "sigma": 2.0},
        # the surrogate's prescreen of 4096 candidates (configuration of the surrogate benchmark)
        {"name": "surrogate_predict", "kind": "predict", "W": 2048, "H": 2048, "P": 4096, "B": 360, "R": 256.0},
        # one training step's sampling, forward and backward on a batch of labelled beams
        {"name": "surrogate_train", "kind": "train", "W": 2048, "H": 2048, "P": 512, "B": 360, "R": 256.0, "N": 4096},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of a listed kind, sizes spread over the range (log-uniform), odd ones included; a
    draw that would cost more than the largest listed case of its kind loses poses."""
    kind = rng.choice(["eval2d", "eval2d", "eval2d", "traj", "update", "eval3d", "eval3d", "encode", "mixed", "predict",
                       "train"])
    W, H = int(_log(rng, 96, 2048)), int(_log(rng, 96, 2048))
    c = {"kind": kind, "W": W, "H": H}
    sigma = round(rng.uniform(1.0, 3.0), 2)
    if kind == "eval2d":
        c |= {"world": rng.choice(["office", "random"]), "P": int(_log(rng, 1, 1024)), "B": int(_log(rng, 24, 720)),
              "R": round(_log(rng, 12, 512), 1), "variant": rng.choice(["exact", "exact", "approx", "uniform"]),
              "sigma": sigma, "band": rng.randint(1, 8), "e0": rng.randint(0, 1)}
        c["P"] = max(1, min(c["P"], int(1024 * 360 * 256 / (c["B"] * c["R"]))))
    elif kind == "traj":
        W, H = int(_log(rng, 96, 1024)), int(_log(rng, 96, 1024))
        c |= {"W": W, "H": H, "world": "office", "T": int(_log(rng, 2, 48)), "S": rng.randint(2, 16),
              "B": int(_log(rng, 24, 181)), "R": round(_log(rng, 16, 128), 1), "sigma": sigma}
    elif kind == "update":
        W, H = int(_log(rng, 96, 1024)), int(_log(rng, 96, 1024))
        c |= {"W": W, "H": H, "world": "office", "P": int(_log(rng, 1, 32)), "B": int(_log(rng, 60, 720)),
              "R": round(_log(rng, 16, 200), 1)}
    elif kind in ("eval3d", "encode"):
        big = kind == "eval3d"
        v = rng.choice(["exact", "exact", "approx", "uniform"])
        c = {"kind": kind, "X": int(_log(rng, 64, 512 if big else 256)), "Y": int(_log(rng, 64, 512 if big else 256)),
             "Z": int(_log(rng, 24, 128 if big else 96)), "P": int(_log(rng, 1, 64 if big else 12)),
             "rw": int(_log(rng, 16, 128 if big else 96)), "rh": int(_log(rng, 16, 128 if big else 96)),
             "R": int(_log(rng, 32, 384 if big else 256)), "variant": v, "reading": rng.randint(0, 1),
             "sigma": 2.0 if rng.random() < 0.5 else sigma, "band": rng.randint(2, 8), "cap": rng.choice([16, 64, 64, 255])}
    elif kind == "mixed":
        c |= {"W": int(_log(rng, 128, 1024)), "H": int(_log(rng, 128, 1024)), "X": int(_log(rng, 64, 192)),
              "Y": int(_log(rng, 64, 192)), "Z": int(_log(rng, 24, 64)), "sets": int(_log(rng, 4, 64)),
              "pmax2": int(_log(rng, 4, 96)), "pmax3": rng.randint(1, 6), "B": int(_log(rng, 60, 360)),
              "rw": rng.randint(16, 64), "rh": rng.randint(16, 64), "rmax2": int(_log(rng, 24, 128)),
              "rmax3": int(_log(rng, 24, 128)), "sigma": sigma}
    elif kind == "predict":
        c |= {"P": int(_log(rng, 1, 4096)), "B": int(_log(rng, 24, 361)), "R": round(_log(rng, 32, 256), 1)}
    else:
        c |= {"P": int(_log(rng, 16, 512)), "B": int(_log(rng, 24, 361)), "R": round(_log(rng, 32, 256), 1),
              "N": int(_log(rng, 128, 4096))}
    return c


# ---- inputs ----------------------------------------------------------------------------------------


def _grid(case, seed):
    """float32 [H][W]: an explored building (walls, free and unknown space), or independent cells."""
    W, H = case["W"], case["H"]
    if case.get("world", "office") == "random":
        return np.random.default_rng(seed).uniform(0.05, 0.95, size=(H, W)).astype(np.float32)
    size = max(W, H)
    return np.ascontiguousarray(synth.office_grid(size, max(8, 400 * size * size // (2048 * 2048)), 0.40, seed)[:H, :W])


def _poses2(grid, n, rng):
    """n poses in free space at any position inside their cell and any yaw."""
    ys, xs = np.nonzero(grid < 0.5)
    if len(xs) == 0:
        ys, xs = np.nonzero(grid >= 0.0)
    i = rng.integers(0, len(xs), n)
    p = np.empty((n, 4), np.int32)
    p[:, 0] = xs[i] * 65536 + rng.integers(0, 65536, n)
    p[:, 1] = ys[i] * 65536 + rng.integers(0, 65536, n)
    a = rng.uniform(0.0, 2.0 * math.pi, n)
    p[:, 2], p[:, 3] = synth.q30(np.cos(a)), synth.q30(np.sin(a))
    return p


def _traj_poses(case, grid, rng):
    """T paths of S states, about two cells apart along a slowly turning heading, kept inside the map."""
    T, S = case["T"], case["S"]
    start = _poses2(grid, T, rng)
    p = np.empty((T, S, 4), np.int32)
    h = rng.uniform(0.0, 2.0 * math.pi, T)
    x, y = start[:, 0] / 65536.0, start[:, 1] / 65536.0
    for s in range(S):
        p[:, s, 0] = np.rint(np.clip(x, 0.5, case["W"] - 0.5) * 65536)
        p[:, s, 1] = np.rint(np.clip(y, 0.5, case["H"] - 0.5) * 65536)
        p[:, s, 2], p[:, s, 3] = synth.q30(np.cos(h)), synth.q30(np.sin(h))
        x, y, h = x + 2.0 * np.cos(h), y + 2.0 * np.sin(h), h + rng.normal(0.0, 0.1, T)
    return p.reshape(T * S, 4)


def _volume(case, seed):
    X, Y, Z = case["X"], case["Y"], case["Z"]
    boxes = max(4, int(round(200 * X * Y * Z / (512 * 512 * 128))))
    return synth.voxel_world(X, Y, Z, n_boxes=boxes, seed=seed, noise_seed=seed + 1)


def _poses3(vox, n, rng):
    Z = vox.shape[0]
    return synth.free_voxel_poses(vox, n, seed=int(rng.integers(1 << 30)), zlo=Z // 4, zhi=max(Z // 4 + 1, 3 * Z // 4))


def _prm(case, **kw):
    base = dict(sigma=case.get("sigma", 2.0), delta_occ=DOCC, delta_emp=DEMP, max_range=float(case.get("R", 64)),
                variant=VARIANTS[case.get("variant", "exact")], trunc_delta=case.get("band", 3),
                uniform_h=case.get("band", 3), e0_mode=case.get("e0", 0), approx_reading=case.get("reading", 0),
                run_cap=case.get("cap", 64))
    base.update(kw)
    return fsmi.Params(**base)


def _store(case):
    """Runs a caller makes room for: one for every second virtual cell."""
    return case["P"] * case["rw"] * case["rh"] * (case["R"] // 2)


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _host(case, seed):
    """The case's inputs as numpy arrays."""
    rng = np.random.default_rng(seed)
    kind, h = case["kind"], {}
    if kind in ("eval2d", "traj", "update", "mixed", "predict", "train"):
        h["grid"] = _grid(case, seed)
        h["dirs"] = synth.beam_dirs_2d(case["B"])
        if kind == "traj":
            h["poses"] = _traj_poses(case, h["grid"], rng)
            h["off"] = (np.arange(case["T"] + 1) * case["S"]).astype(np.int32)
        elif kind != "mixed":
            h["poses"] = _poses2(h["grid"], case["P"], rng)
    if kind == "update":  # measured ranges: hits at all distances, one beam in five without return
        z = rng.uniform(0.5, case["R"], (case["P"], case["B"])).astype(np.float32)
        z[rng.random(z.shape) < 0.2] = np.inf
        h["ranges"] = z
    if kind in ("eval3d", "encode", "mixed"):
        h["vox"] = _volume(case, seed)
        h["dirs3"] = synth.pinhole_dirs(case["rw"], case["rh"], 90.0)
        if kind != "mixed":
            h["poses3"] = _poses3(h["vox"], case["P"], rng)
    if kind == "mixed":
        sets, n2, n3 = [], 0, 0
        rng = np.random.default_rng(case["sets"] * 1000 + case["B"])  # the same sets for every seed: one output size
        for k in range(case["sets"]):
            three = k % 2 == 1
            r = float(np.exp(rng.uniform(math.log(8), math.log(case["rmax3" if three else "rmax2"]))))
            if three:
                P = int(rng.integers(1, case["pmax3"] + 1))
                sets.append((fsmi.SET_3D, n3, P, 0, case["rw"] * case["rh"], math.floor(r), 0))
                n3 += P
            else:
                P = int(rng.integers(1, case["pmax2"] + 1))
                sets.append((fsmi.SET_2D, n2, P, 0, case["B"], round(r, 1)))
                n2 += P
        rng = np.random.default_rng(seed + 1)
        h |= {"sets": sets, "poses": _poses2(h["grid"], max(n2, 1), rng), "poses3": _poses3(h["vox"], max(n3, 1), rng)}
    if kind == "train":
        h["ids"] = rng.integers(0, case["P"] * case["B"], case["N"]).astype(np.int32)
        h["labels"] = rng.normal(0.0, 1.0, case["P"] * case["B"]).astype(np.float32)
    return h


def prepare(case, seed):
    h = _host(case, seed)
    kind = case["kind"]
    s = {"case": case, **{k: _cuda(v) for k, v in h.items() if isinstance(v, np.ndarray)}}
    if kind in ("eval2d", "eval3d"):
        s["prm"] = _prm(case)
    elif kind == "traj":
        s["prm"] = _prm(case)
        s["ws"] = torch.empty(fsmi.trajectory_workspace_size(case["W"], case["H"], case["T"]), dtype=torch.uint8,
                              device="cuda")
    elif kind == "update":
        s["prm"] = _prm(case)
        s["map"] = torch.empty_like(s["grid"])
    elif kind == "encode":
        # a capacity of exactly the runs of these views, as a first counting call reports it
        s["prm"] = _prm(case)
        off, _, _ = fsmi.rle_encode_3d(s["vox"], s["poses3"], s["dirs3"], s["prm"], 0)
        s["capacity"] = int(off[-1].item())
        fsmi.device_status()
        # where the caller keeps the runs, sized before they are known
        s["run_o"] = torch.zeros(_store(case), dtype=torch.float32, device="cuda")
        s["run_len"] = torch.zeros(_store(case), dtype=torch.uint8, device="cuda")
    elif kind == "mixed":
        s["sets"], s["nitems"] = fsmi.make_sets(h["sets"], "cuda")
        s["volumes"] = fsmi.make_volumes([s["vox"]], "cuda")
        s["prm2"] = _prm(case, max_range=float(case["rmax2"]))
        s["prm3"] = _prm(case, max_range=float(case["rmax3"]))
    elif kind in ("predict", "train"):
        s["net"] = surrogate.Surrogate(seed=seed)
        # the trained biases are not zero
        s["net"].params.add_(torch.from_numpy(_bias_noise(seed)).cuda())
        fsmi.surrogate_cast(s["net"].params, s["net"].wbf16)
        if kind == "train":
            N = case["N"]
            s["x"] = torch.empty((N, fsmi.SURR_L, 2), dtype=torch.bfloat16, device="cuda")
            s["y"] = torch.empty(N, dtype=torch.float32, device="cuda")
            s["pred"] = torch.empty(N, dtype=torch.float32, device="cuda")
            s["ws"] = torch.empty(fsmi.surrogate_workspace_size(0, N), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "eval2d":
        return fsmi.eval_2d(s["grid"], s["poses"], s["dirs"], s["prm"])
    if kind == "traj":
        return fsmi.eval_trajectories_2d(s["grid"], s["poses"], s["off"], s["dirs"], s["prm"], ws=s["ws"])
    if kind == "update":  # the prior map is kept: each pass updates a copy of it
        return fsmi.update_map_2d(s["map"].copy_(s["grid"]), s["poses"], s["dirs"], s["ranges"], s["prm"])
    if kind == "eval3d":
        return fsmi.eval_3d(s["vox"], s["poses3"], s["dirs3"], s["prm"])
    if kind == "encode":
        off, ro, rl = fsmi.rle_encode_3d(s["vox"], s["poses3"], s["dirs3"], s["prm"], s["capacity"])
        s["run_o"][:s["capacity"]].copy_(ro)
        s["run_len"][:s["capacity"]].copy_(rl)
        return [off, s["run_o"], s["run_len"], fsmi.eval_rle(off, ro, rl, s["prm"])]
    if kind == "mixed":
        return fsmi.eval_mixed(s["sets"], s["nitems"], grid=s["grid"], poses2=s["poses"], dirs2=s["dirs"],
                               prm2=s["prm2"], volumes=s["volumes"], poses3=s["poses3"], dirs3=s["dirs3"],
                               prm3=s["prm3"])
    net = s["net"]
    if kind == "predict":
        return net.predict(s["grid"], s["poses"], s["dirs"], max_range=case["R"])
    # as Surrogate.train issues a step, up to the gradient
    fsmi.profiles_2d(s["grid"], s["poses"], s["dirs"], beam_ids=s["ids"], out=s["x"], max_range=case["R"])
    fsmi.gather_rows(s["labels"].view(torch.int32).view(-1, 1), s["ids"], out=s["y"].view(torch.int32).view(-1, 1))
    fsmi.surrogate_loss_grad(net.params, net.wbf16, s["x"], s["y"], net.grad, net.loss, pred=s["pred"], ws=s["ws"])
    return [net.loss, net.grad, s["pred"]]


def work(case):
    """Bytes: every input read once and every output written once. Operations: per visited cell the gains
    and prefixes, per pair of cells within the noise kernel's reach the pair term; the network's
    multiply-adds. Beams are taken to reach their range or, on average, half the map."""
    kind = case["kind"]
    prof = lambda r, w, h: min(r, 0.5 * (w + h) / 2)  # noqa: E731  cells along a beam that may leave the map
    b = f = 0.0
    if kind in ("eval2d", "traj", "update"):
        nb = case["B"] * (case["T"] * case["S"] if kind == "traj" else case["P"])
        n = 1.27 * prof(case["R"], case["W"], case["H"])
        b = 4.0 * min(case["W"] * case["H"], nb * n) + 4.0 * nb
        v = case.get("variant", "exact")
        band = 2 * 5.7 * case.get("sigma", 2.0) * 1.27 if v == "exact" else 2 * case.get("band", 0) + 2
        f = nb * n * (30.0 + (0 if kind == "update" else 4.0 if v == "uniform" else 12.0 * band))
        if kind == "update":
            b += 4.0 * case["W"] * case["H"] + 4.0 * nb
    elif kind in ("eval3d", "encode"):
        nb = case["P"] * case["rw"] * case["rh"]
        n = prof(case["R"], case["X"], case["Y"])
        K = 2 * (case["band"] if case["variant"] == "uniform" else math.ceil(7.45 * case["sigma"])) + 1
        b = 4.0 * min(case["X"] * case["Y"] * case["Z"], nb * n) + 4.0 * nb + (5.0 * nb * n / 5 if kind == "encode" else 0)
        f = nb * n * (60.0 + 2.0 * K)
    elif kind == "mixed":
        n2 = case["sets"] / 2 * case["pmax2"] / 2 * case["B"]
        n3 = case["sets"] / 2 * case["pmax3"] / 2 * case["rw"] * case["rh"]
        r2, r3 = (case["rmax2"] - 8) / math.log(case["rmax2"] / 8), (case["rmax3"] - 8) / math.log(case["rmax3"] / 8)
        r3 = prof(r3, case["X"], case["Y"])
        b = 4.0 * (min(case["W"] * case["H"], n2 * r2) + min(case["X"] * case["Y"] * case["Z"], n3 * r3) + n2 + n3)
        f = n2 * r2 * 1.27 * (30 + 12 * 2 * 5.7 * case["sigma"] * 1.27) + n3 * r3 * (60 + 4 * math.ceil(7.45 * case["sigma"]))
    else:
        macs = 128 * 32 * 6 + 64 * 32 * 96 + 32 * 32 * 96 + 1024 * 256 + 256
        nb = case["P"] * case["B"] if kind == "predict" else case["N"]
        b = 4.0 * min(case["W"] * case["H"], 256.0 * nb) + 4.0 * nb + 2.0 * fsmi.SURR_NPARAMS
        f = 2.0 * macs * nb
        if kind == "train":
            # the pre-activations are part of the documented result (they stay in the workspace)
            b += 4.0 * nb * (128 * 32 + 64 * 32 + 32 * 32 + 256) + 4.0 * fsmi.SURR_NPARAMS
            f *= 3
    return {"bytes": b, "flops": f}


# ---- the results in 64 bits -------------------------------------------------------------------------


def _bias_noise(seed):
    g, out = np.random.default_rng(seed + 5), []
    for name, shape in surrogate.LAYOUT:
        n = int(np.prod(shape))
        out.append(g.uniform(-0.05, 0.05, n).astype(np.float32) if name.startswith("b") else np.zeros(n, np.float32))
    return np.concatenate(out)


def _gain(delta, o):
    """f(delta, r): the divergence of the posterior from the prior o of a cell."""
    delta = float(np.float32(delta))
    post = o * delta / (o * delta + 1.0 - o)
    return torch.special.xlogy(post, post / o.clamp_min(1e-300)) + \
        torch.special.xlogy(1.0 - post, (1.0 - post) / (1.0 - o).clamp_min(1e-300))


def _beam_dirs(pose, u):
    """Beam directions (Q30) of sensor-frame directions u under poses, int64 [n][2]."""
    c, s = pose[:, 2], pose[:, 3]
    dx = (c * u[:, 0] - s * u[:, 1] + (1 << 29)) >> 30
    dy = (s * u[:, 0] + c * u[:, 1] + (1 << 29)) >> 30
    return dx, dy


def _trace(W, H, pose, u, rfix):
    """Cells of n beams in order, by exact integer comparison of the crossings. Returns (ids int64
    [n][L], l float64 [n][L+1] with l[:, j >= count] the end distance, count [n], by_range [n])."""
    dx, dy = _beam_dirs(pose, u)
    ox, oy = pose[:, 0], pose[:, 1]
    cx = (ox >> 16) - ((dx < 0) & (ox & 0xFFFF == 0)).long()
    cy = (oy >> 16) - ((dy < 0) & (oy & 0xFFFF == 0)).long()
    xm = dx.abs() >= dy.abs()
    pick = lambda a, b: torch.where(xm, a, b)  # noqa: E731
    dM, dm, oM, om, cM, cm = pick(dx, dy), pick(dy, dx), pick(ox, oy), pick(oy, ox), pick(cx, cy), pick(cy, cx)
    dimM, dimm = pick(torch.full_like(dx, W), torch.full_like(dx, H)), pick(torch.full_like(dx, H), torch.full_like(dx, W))
    aM, am = dM.abs(), dm.abs()
    sM, sm = torch.where(dM > 0, 1, -1), torch.where(dm > 0, 1, -1)
    nM0 = torch.where(sM > 0, ((cM + 1) << 16) - oM, oM - (cM << 16))
    nm0 = torch.where(sm > 0, ((cm + 1) << 16) - om, om - (cm << 16))
    limM, limm = ((rfix * aM - 1) >> 30) + 1, ((rfix * am - 1) >> 30) + 1  # numerators below these enter before R
    K = int(rfix.max().item() >> 16) + 3
    k = torch.arange(-1, K, device=pose.device)[None, :]
    c1 = lambda v: v[:, None]  # noqa: E731
    nM = c1(nM0) + k * 65536                     # the crossing that opens interval k (k >= 0)
    has = c1(am) > 0
    amc, aMc = c1(am), c1(aM).clamp_min(1)
    num = nM * amc - c1(nm0) * aMc
    i = torch.where((k >= 0) & has & (num >= 0), torch.div(num, aMc << 16, rounding_mode="floor") + 1, 0)
    nm = c1(nm0) + i * 65536                     # the next minor crossing
    inner = has & (nm * aMc < (nM + 65536) * amc)  # strictly inside the interval
    lamM, lamm = nM.double() * 16384.0 / aMc, nm.double() * 16384.0 / amc.clamp_min(1)
    lamM = torch.where(k < 0, 0.0, lamM)
    a_M, a_m = c1(cM) + c1(sM) * (k + 1), c1(cm) + c1(sm) * i
    okM = ((k < 0) | (nM < c1(limM))) & (a_M >= 0) & (a_M < c1(dimM)) & (a_m >= 0) & (a_m < c1(dimm))
    b_m = a_m + c1(sm)
    okm = (nm < c1(limm)) & (b_m >= 0) & (b_m < c1(dimm)) & (a_M >= 0) & (a_M < c1(dimM))
    rangeM, rangem = (k >= 0) & (nM >= c1(limM)), nm >= c1(limm)
    two = lambda p, q: torch.stack([p, q], 2).reshape(p.shape[0], -1)  # noqa: E731
    exist = two(torch.ones_like(inner), inner)
    ok = two(okM, okm)
    xid = lambda M, m: torch.where(c1(xm), m * W + M, M * W + m)  # noqa: E731
    ids, lam = two(xid(a_M, a_m), xid(a_M, b_m)), two(lamM, lamm)
    by_rng = two(rangeM.expand_as(inner), rangem)
    order = torch.argsort((~exist).to(torch.uint8), dim=1, stable=True)  # crossings that exist, in order
    exist, ok, ids, lam, by_rng = (v.gather(1, order) for v in (exist, ok, ids, lam, by_rng))
    ok = ok & exist
    count = ok.long().cumprod(1).sum(1)
    count = torch.where((dx == 0) & (dy == 0), 0, count)
    last = count.clamp_max(ok.shape[1] - 1)[:, None]
    R = rfix.double() / 65536.0
    ended = by_rng.gather(1, last)[:, 0]
    end = torch.where(ended, R, torch.minimum(lam.gather(1, last)[:, 0], R))
    L = max(1, int(count.max().item()))
    j = torch.arange(L + 1, device=pose.device)[None, :]
    lam = torch.where(j < count[:, None], lam[:, :L + 1], end[:, None])
    return torch.where(j[:, :L] < count[:, None], ids[:, :L], 0), lam, count, ended & (count > 0)


def _phi(x):
    return 0.5 * torch.special.erfc(-x * 0.7071067811865476)


def _beam_mi(o, fo, fe, l, count, case, variant, band, e0):
    """Pair sums of Section 3 in 64 bits: o, f_occ, f_emp [n][L] (zero beyond count), l [n][L+1]."""
    n, L = o.shape
    keep = torch.arange(L, device=o.device)[None, :] < count[:, None]
    o = torch.where(keep, o, 0.0)
    q = torch.cumprod(1.0 - o, 1)
    P = o * torch.cat([torch.ones_like(q[:, :1]), q[:, :-1]], 1)
    pe0 = q[:, -1]
    S = torch.cumsum(torch.where(keep, fe, 0.0), 1)
    C = torch.where(keep, torch.cat([torch.zeros_like(S[:, :1]), S[:, :-1]], 1) + fo, 0.0)
    mi = torch.zeros(n, dtype=torch.float64, device=o.device)
    none = torch.zeros_like(pe0)
    if variant == "uniform":
        D = torch.cat([torch.zeros_like(C[:, :1]), torch.cumsum(C, 1)], 1)  # D[:, k] = C_1 + .. + C_k
        j = torch.arange(1, L + 1, device=o.device)[None, :]
        hi = torch.minimum(count[:, None], j + band)
        lo = (j - band - 1).clamp_min(0)
        mi = (P * (D.gather(1, hi) - D.gather(1, lo.expand_as(hi)))).sum(1) / (2 * band + 1)
        if e0:
            mi = mi + pe0 * D.gather(1, torch.minimum(count, torch.full_like(count, band))[:, None])[:, 0] / (2 * band + 1)
        return torch.where(count > 0, mi, none)
    sigma = float(np.float32(case["sigma"]))
    mu = 0.5 * (l[:, :-1] + l[:, 1:])
    W = band if variant == "approx" else int(math.ceil(9.0 * sigma * 1.5)) + 3  # cells within 9 sigma
    pad = torch.nn.functional.pad
    lp, Cp = torch.cat([l[:, :1].expand(n, W), l, l[:, -1:].expand(n, W)], 1), pad(C, (W, W))
    T = _phi((lp[:, 0:L] - mu) / sigma)
    for d in range(2 * W + 1):  # cell j + d - W
        nxt = _phi((lp[:, d + 1:d + 1 + L] - mu) / sigma)
        mi = mi + (P * Cp[:, d:d + L] * (nxt - T)).sum(1)
        T = nxt
    if e0:  # the no-return event, centred half a cell before the first boundary
        kmax = min(L, band) if variant == "approx" else L
        x = _phi((l[:, :kmax + 1] - (l[:, :1] - 0.5)) / sigma)
        mi = mi + pe0 * (C[:, :kmax] * (x[:, 1:] - x[:, :-1])).sum(1)
    return torch.where(count > 0, mi, none)


def _scan(grid, pose, u, rfix, case, variant, band, e0, stamp=None, state=None):
    """Exact per-beam MI for beams (pose[i], u[i]) with ranges rfix (Q16)."""
    H, W = grid.shape
    flat = grid.reshape(-1).double()
    ids, l, count, _ = _trace(W, H, pose, u, rfix)
    o = flat[ids]
    fo, fe = _gain(DOCC, o), _gain(DEMP, o)
    if stamp is not None:
        dead = stamp.gather(1, ids) < state[:, None] if stamp.dim() == 2 else stamp[ids] < state[:, None]
        fo, fe = fo.masked_fill(dead, 0.0), fe.masked_fill(dead, 0.0)
    return _beam_mi(o, fo, fe, l, count, case, variant, band, e0)


def _q16(r):
    return int(np.rint(float(np.float32(r)) * 65536.0))


def _pairs(poses, dirs, lo, hi):
    """Poses and directions of the flat beams lo .. hi - 1 (beam = pose * ndir + direction)."""
    b = torch.arange(lo, hi, device=poses.device)
    return poses[b // dirs.shape[0]].long(), dirs[b % dirs.shape[0]].long()


def _chunks(n, size):
    return [(a, min(n, a + size)) for a in range(0, n, size)]


def _sample3(vox, pose, u, nsamp):
    """Values of the virtual cells of n rays, float64 [n][nsamp], and their counts."""
    Z, Y, X = vox.shape
    i = 2 * torch.arange(nsamp, device=vox.device)[None, :] + 1
    idx, inside = None, None
    for a, dim, stride in ((0, X, 1), (1, Y, X), (2, Z, X * Y)):
        d = (pose[:, 3 + 3 * a] * u[:, 0] + pose[:, 4 + 3 * a] * u[:, 1] + pose[:, 5 + 3 * a] * u[:, 2] + (1 << 29)) >> 30
        p = ((pose[:, a] << 15)[:, None] + i * d[:, None]) >> 31
        ok = (p >= 0) & (p < dim)
        p = p.clamp(0, dim - 1) * stride
        idx, inside = (p, ok) if idx is None else (idx + p, inside & ok)
    count = inside.long().cumprod(1).sum(1)
    return vox.reshape(-1)[idx], count


def _runs(v, count, cap):
    """First virtual cell of each cell's run, [n][L] (runs of equal values split every cap cells)."""
    n, L = v.shape
    j = torch.arange(L, device=v.device)[None, :].expand(n, L)
    new = torch.ones_like(v, dtype=torch.bool)
    new[:, 1:] = v[:, 1:] != v[:, :-1]
    span = torch.where(new, j, 0).cummax(1).values
    return span + (j - span) // cap * cap


def _ray_mi(v, count, case, variant, start):
    """Theorems 3, 5 and 6 per virtual cell, in 64 bits. start: each cell's run's first cell."""
    n, L = v.shape
    j = torch.arange(L, device=v.device)[None, :]
    keep = j < count[:, None]
    o = torch.where(keep, v.double(), 0.0)
    q = torch.cumprod(1.0 - o, 1)
    P = o * torch.cat([torch.ones_like(q[:, :1]), q[:, :-1]], 1)
    S = torch.cumsum(torch.where(keep, _gain(DEMP, o), 0.0), 1)
    C = torch.where(keep, torch.cat([torch.zeros_like(S[:, :1]), S[:, :-1]], 1) + _gain(DOCC, o), 0.0)
    sigma, band = float(np.float32(case["sigma"])), case.get("band", 0)
    K = band if variant == "uniform" else int(math.ceil(9.0 * sigma))
    lo, hi = j - K, j + K + 1
    if variant == "approx" and case["reading"] == 1:
        K = min(K, band)
    elif variant == "approx":  # Theorem 5's kept pairs: whole runs within Delta of one another
        last = (count - 1).clamp_min(0)[:, None]
        cut = keep & torch.cat([start[:, 1:] != start[:, :-1], torch.ones_like(keep[:, :1])], 1)
        stop = torch.where(cut | (j == last), j + 1, 2 * L).flip(1).cummin(1).values.flip(1)
        lo = torch.maximum(start.gather(1, (j - band).clamp_min(0).expand(n, L)), start - band)
        hi = torch.minimum(stop + band, stop.gather(1, torch.minimum(j + band, last).expand(n, L)))
    Cp = torch.nn.functional.pad(C, (K, K))
    mi = torch.zeros(n, dtype=torch.float64, device=v.device)
    for d in range(-K, K + 1):
        g = 1.0 / (2 * band + 1) if variant == "uniform" else \
            math.exp(-d * d / (2.0 * sigma * sigma)) / (math.sqrt(2.0 * math.pi) * sigma)
        t = P * Cp[:, K + d:K + d + L]
        if variant == "approx" and case["reading"] == 0:
            t = t * ((j + d >= lo) & (j + d < hi))
        mi = mi + g * t.sum(1)
    return mi


def _net(theta):
    w, at = {}, 0
    for name, shape in surrogate.LAYOUT:
        n = int(np.prod(shape))
        t = theta[at:at + n]
        w[name] = (t.bfloat16() if name.startswith("W") else t).double().reshape(shape)
        at += n
    return w


def _forward(w, x):
    """The network on profiles x [n][256][2], 64 bits."""
    a = x
    for k in (1, 2, 3):
        n, Lin, ci = a.shape
        p = torch.nn.functional.pad(a, (0, 0, 1, 1))
        cols = torch.cat([p[:, t:t + Lin:2] for t in range(3)], 2)
        a = torch.relu(cols.reshape(-1, 3 * ci) @ w["W%d" % k].reshape(32, -1).T + w["b%d" % k]).reshape(n, Lin // 2, 32)
    h = torch.relu(a.reshape(a.shape[0], 1024) @ w["W4"].T + w["b4"])
    return h @ w["W5"] + w["b5"][0]


def _profile(grid, pose, u, R):
    """Profiles [n][256][2] of beams, BF16 values in 64 bits."""
    H, W = grid.shape
    dx, dy = _beam_dirs(pose, u)
    i = 2 * torch.arange(fsmi.SURR_L, device=grid.device)[None, :] + 1
    px, py = ((pose[:, 0] << 15)[:, None] + i * dx[:, None]) >> 31, ((pose[:, 1] << 15)[:, None] + i * dy[:, None]) >> 31
    ok = (px >= 0) & (px < W) & (py >= 0) & (py < H) & (i * 0.5 < R)
    o = grid[py.clamp(0, H - 1), px.clamp(0, W - 1)].bfloat16().double()
    return torch.stack([torch.where(ok, o, 0.0), ok.double()], 2)


def exact(case, seed):
    h = _host(case, seed)
    kind, dev = case["kind"], "cuda" if torch.cuda.is_available() else "cpu"
    t = {k: torch.from_numpy(np.ascontiguousarray(v)).to(dev) for k, v in h.items() if isinstance(v, np.ndarray)}
    full = lambda n, r: torch.full((n,), r, dtype=torch.int64, device=dev)  # noqa: E731
    if kind == "eval2d":
        nb, out = case["P"] * case["B"], []
        for a, b in _chunks(nb, 16384):
            p, u = _pairs(t["poses"], t["dirs"], a, b)
            out.append(_scan(t["grid"], p, u, full(b - a, _q16(case["R"])), case, case["variant"], case["band"], case["e0"]))
        return torch.cat(out).reshape(case["P"], case["B"])
    if kind == "traj":
        B, S, beams = case["B"], case["S"], []
        cells = case["W"] * case["H"]
        for k in range(case["T"]):
            p, u = _pairs(t["poses"][k * S:(k + 1) * S], t["dirs"], 0, S * B)
            st = torch.arange(S * B, device=dev) // B
            ids, _, count, _ = _trace(case["W"], case["H"], p, u, full(S * B, _q16(case["R"])))
            m = torch.arange(ids.shape[1], device=dev)[None, :] < count[:, None]
            stamp = torch.full((cells,), 1 << 20, dtype=torch.int64, device=dev)
            stamp.scatter_reduce_(0, ids[m], st[:, None].expand_as(ids)[m], "amin")
            beams.append(_scan(t["grid"], p, u, full(S * B, _q16(case["R"])), case, "exact", 0, 0, stamp, st))
        beam = torch.cat(beams).reshape(-1, B)
        state = beam.sum(1)
        return [beam, state, state.reshape(case["T"], S).sum(1)]
    if kind == "update":
        z = t["ranges"].reshape(-1).double()
        top = _q16(case["R"])
        hit = torch.isfinite(z) & (torch.round(z.clamp(max=1e6) * 65536.0).long() < top)
        rfix = torch.where(hit, torch.round(z.clamp(max=1e6) * 65536.0).long(), top)
        add = torch.zeros(case["W"] * case["H"], dtype=torch.float64, device=dev)
        lo, le = math.log(float(np.float32(DOCC))), math.log(float(np.float32(DEMP)))
        for a, b in _chunks(z.numel(), 16384):
            p, u = _pairs(t["poses"], t["dirs"], a, b)
            ids, _, count, by_range = _trace(case["W"], case["H"], p, u, rfix[a:b])
            j = torch.arange(ids.shape[1], device=dev)[None, :]
            m = j < count[:, None]
            occ = (hit[a:b] & by_range)[:, None] & (j == count[:, None] - 1)
            add.index_add_(0, ids[m], torch.where(occ, lo, le)[m].double())
        o = t["grid"].reshape(-1).double()
        return torch.sigmoid(torch.log(o) - torch.log1p(-o) + add).reshape(t["grid"].shape)
    if kind in ("eval3d", "encode"):
        nb, out, runs = case["P"] * case["rw"] * case["rh"], [], []
        for a, b in _chunks(nb, 16384):
            p, u = _pairs(t["poses3"], t["dirs3"], a, b)
            v, count = _sample3(t["vox"], p, u, case["R"])
            start = _runs(v, count, case["cap"])
            out.append(_ray_mi(v, count, case, case["variant"], start))
            if kind == "encode":
                j = torch.arange(v.shape[1], device=dev)[None, :]
                runs.append(v[(j < count[:, None]) & (start == j)].double())
        mi = torch.cat(out)
        if kind == "eval3d":
            return mi.reshape(case["P"], -1)
        kept, runs = torch.zeros(_store(case), dtype=torch.float64, device=dev), torch.cat(runs)
        kept[:runs.numel()] = runs
        return [None, kept, None, mi]
    if kind == "mixed":
        out = []
        for st in h["sets"]:
            k, po, P, do, nd, r = st[:6]
            for a, b in _chunks(P * nd, 16384):
                if k == fsmi.SET_2D:
                    p, u = _pairs(t["poses"][po:po + P], t["dirs"], a, b)
                    out.append(_scan(t["grid"], p, u, full(b - a, _q16(r)), case, "exact", 0, 0))
                else:
                    p, u = _pairs(t["poses3"][po:po + P], t["dirs3"], a, b)
                    v, count = _sample3(t["vox"], p, u, int(r))
                    out.append(_ray_mi(v, count, case, "exact", None))
        return torch.cat(out)
    w = _net(torch.from_numpy(surrogate.init_params(seed) + _bias_noise(seed)).to(dev))
    if kind == "predict":
        out = []
        for a, b in _chunks(case["P"] * case["B"], 32768):
            p, u = _pairs(t["poses"], t["dirs"], a, b)
            out.append(_forward(w, _profile(t["grid"], p, u, case["R"])))
        return torch.cat(out)
    ids = t["ids"].long()
    x = _profile(t["grid"], t["poses"][ids // case["B"]].long(), t["dirs"][ids % case["B"]].long(), case["R"])
    for v in w.values():
        v.requires_grad_(True)
    pred = _forward(w, x)
    loss = ((pred - t["labels"][ids].double()) ** 2).mean()
    loss.backward()
    grad = torch.cat([w[name].grad.reshape(-1) for name, _ in surrogate.LAYOUT])
    return [loss.detach().reshape(1), grad, pred.detach()]
